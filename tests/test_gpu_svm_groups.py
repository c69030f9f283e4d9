"""Tensor-core window scores where its work cut can go wrong.

The kernel walks items of 26 window columns, four at a time per SM, and cuts small
plans into pieces of a few window rows. Sizes: one column, one short of, at and one
past a group, two groups and one; one row up to one past the 64-row limit; a flat
level, whose blocks put all 256 counts into one LBP bin (the last table entry).
Bar: |gpu - ref| <= 1e-4 (|b| + sum |w x|), the score bar of the other tests; the
scores do not depend on the item height at all.
"""
import os

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("cols,rows,flat", [(1, 1, False), (25, 2, False), (26, 17, False), (27, 65, False),
                                            (53, 3, False), (27, 3, True)])
def test_scores_at_group_edges(cols, rows, flat):
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    w, b = d["w"], float(d["b"])
    W, H = 8 * (cols + 7) + 3, 8 * (rows + 15) + 5
    L = np.full((H, W), 90, np.uint8) if flat else synth.random_image(W, H, 60 + cols)
    hog, lbp = oracle.hog_cells(L).astype(np.float32), oracle.lbp_cells(L)
    feat = oracle.block_features(hog.astype(np.float64), lbp)
    ref = oracle.scores(feat, w, b)
    assert ref.shape == (rows, cols)
    scale = abs(b) + oracle.scores(feat, np.abs(w), 0.0)
    hc, wc = rows + 15, cols + 7
    pitch = (wc + 15) // 16 * 16
    hp, lp = np.zeros((9, hc, pitch), np.float32), np.zeros((59, hc, pitch), np.uint8)
    hp[:, :, :wc], lp[:, :, :wc] = hog.transpose(2, 0, 1), lbp.transpose(2, 0, 1)
    hd, ld = torch.from_numpy(hp).cuda(), torch.from_numpy(lp).cuda()
    det = pd.Detector(w, b, max_frames=1, max_width=W, max_height=H)
    try:
        got = []
        for item_rows in (64, 8):
            pd.pd_set_tuning(det.h, 8, item_rows)
            out = torch.full((rows, cols), float("nan"), device="cuda")
            pd.pd_window_scores(det.h, hd, hc * pitch, ld, hc * pitch, pitch, wc, hc, out)
            torch.cuda.synchronize()
            got.append(out.cpu().numpy())
    finally:
        det.close()
    assert np.array_equal(got[0], got[1])
    assert np.all(np.abs(got[0] - ref) <= 1e-4 * scale)
