"""LBP cell counts where the bit-plane counting can go wrong: exact against the oracle.

Images of few grey values make every one of the 256 codes appear, ties included. Sizes:
one cell, one cell short of, at and past a 15-cell strip, cells cut by the right and
bottom edges, and more than 32 cell rows (two strips on a tall level). The counts of the
cell-major layout, which only the whole path uses, are checked through its scores against
the FP32 kernel's, which reads planes (both within 1e-4 of the oracle's scale, so within
2e-4 of each other).
"""
import os

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _image(W, H, seed, values):
    return (np.random.default_rng(seed).integers(0, values, size=(H, W)) * (250 // values)).astype(np.uint8)


@pytest.mark.parametrize("W,H,values", [(8, 8, 3), (112, 16, 2), (120, 24, 4), (121, 31, 2), (128, 17, 5),
                                        (247, 290, 3), (19, 264, 2)])
def test_counts_are_exact(W, H, values):
    img = _image(W, H, W + H, values)
    ref = oracle.lbp_cells(img)
    hc, wc = ref.shape[:2]
    pitch = (wc + 15) // 16 * 16
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    det = pd.Detector(d["w"], float(d["b"]), max_frames=1, max_width=max(W, 64), max_height=max(H, 128))
    try:
        hog = torch.zeros(9 * hc * pitch, device="cuda")
        lbp = torch.zeros(59 * hc * pitch, dtype=torch.uint8, device="cuda")
        pd.pd_cell_features(det.h, torch.from_numpy(img).cuda(), hog, hc * pitch, lbp, hc * pitch, pitch)
        torch.cuda.synchronize()
    finally:
        det.close()
    got = lbp.cpu().numpy().reshape(59, hc, pitch)[:, :, :wc].transpose(1, 2, 0)
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("W,H,values", [(64, 128, 3), (257, 301, 2)])
def test_cell_major_counts_give_the_planes_scores(W, H, values):
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    frame = torch.from_numpy(_image(W, H, W, values)).cuda()
    maps = []
    for flags in (0, pd.PD_FLAG_SVM_FP32):
        det = pd.Detector(d["w"], float(d["b"]), max_frames=1, max_width=W, max_height=H, flags=flags)
        try:
            det.detect([frame])
            assert det.sync() in (pd.PD_OK, pd.PD_EOVERFLOW)
            maps.append(torch.cat([m.reshape(-1) for m in det.score_maps(0)]).cpu().numpy().astype(np.float64))
        finally:
            det.close()
    scale = abs(float(d["b"])) + np.abs(d["w"].astype(np.float64)).sum()  # features are at most 1
    assert np.all(np.abs(maps[0] - maps[1]) <= 2e-4 * scale)
