"""Pyramid kernel on both tile heights (a plan of many tiles takes tiles twice as
tall): every level byte for byte the oracle's, at frame heights where the last
tall tile holds one row, one half or all of its rows."""
import os

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


# 128 x 32 source tiles: 3 x 3 and 21 x 21 = 441 (short), 22 x 21, 21 x 22, 23 x 22 and 30 x 40 (tall)
@pytest.mark.parametrize("W,H", [(300, 65), (2688, 672), (2689, 672), (2688, 673), (2817, 704), (3840, 1279)])
@pytest.mark.parametrize("groups", [4, 8, 16])
def test_levels_equal_the_oracle(W, H, groups):
    from paper_1611_01642_gb300 import build as bld
    bld.build()
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    img = synth.random_image(W, H, W + H, smooth=False)
    dims = [(W, H), (W * 3 // 2, H * 3 // 2), (int(W / 1.05), int(H / 1.05)), (W // 3, H // 3), (W // 13, H // 5), (17, 1)]
    pitches = [(w + 15) // 16 * 16 for w, _ in dims]
    offs = np.concatenate([[0], np.cumsum([p * h for p, (_, h) in zip(pitches, dims)])]).astype(np.int64)
    out = torch.zeros((int(offs[-1]),), dtype=torch.uint8, device="cuda")
    h = pd.Detector(d["w"], float(d["b"]), max_frames=1, max_width=W, max_height=max(H, 128))
    try:
        pd.pd_set_tuning(h.h, groups, 64)
        pd.pd_resize_levels(h.h, torch.from_numpy(img).cuda(), dims, out, offs[:-1].tolist(), pitches)
        torch.cuda.synchronize()
    finally:
        h.close()
    got = out.cpu().numpy()
    for (w, hh), p, o in zip(dims, pitches, offs):
        lv = got[o:o + p * hh].reshape(hh, p)[:, :w]
        assert np.array_equal(lv, oracle.resize(img, w, hh)), (w, hh)
