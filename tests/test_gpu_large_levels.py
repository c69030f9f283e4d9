"""Window scores of levels far larger than the handle's own, on the tensor cores: taller than a
grid has blocks, with more work items than the handle's descriptor block holds. Any part of
the score map is, bit for bit, that of the part of the level under it alone (a score is one
sum in one order, whatever the level it lies in)."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _planes(cx, cy, seed):
    """Random HOG and LBP planes [planes][cy][pitch]; counts 0..64."""
    pitch = (cx + 15) // 16 * 16
    g = torch.Generator(device="cuda").manual_seed(seed)
    hog = torch.rand(9, cy, pitch, generator=g, device="cuda").mul_(900.0)
    lbp = torch.randint(0, 65, (59, cy, pitch), generator=g, device="cuda", dtype=torch.uint8)
    return hog, lbp, pitch


def _part(det, hog, lbp, pitch, x0, y0, cx, cy):
    """Scores of the cells [x0, x0 + cx) x [y0, y0 + cy) as a level of their own (x0 a multiple of 16)."""
    plane = hog.shape[1] * pitch
    at = y0 * pitch + x0
    out = torch.full((cy - 15, cx - 7), float("nan"), device="cuda")
    pd.pd_window_scores(det.h, hog.reshape(-1)[at:], plane, lbp.reshape(-1)[at:], plane, pitch, cx, cy, out)
    return out


def _check(cx, cy, parts):
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    hog, lbp, pitch = _planes(cx, cy, cx + cy)
    det = pd.Detector(d["w"], float(d["b"]), max_frames=1, max_width=64, max_height=128)
    try:
        full = _part(det, hog, lbp, pitch, 0, 0, cx, cy)
        for x0, y0, w, h in parts:
            part = _part(det, hog, lbp, pitch, x0, y0, w, h)
            assert torch.equal(part, full[y0:y0 + h - 15, x0:x0 + w - 7]), (x0, y0)
    finally:
        torch.cuda.synchronize()
        det.close()


def test_taller_than_a_grid():
    _check(20, 65600, [(0, 0, 20, 90), (0, 65480, 20, 120), (0, 65520, 20, 80)])


def test_more_items_than_the_descriptor_block_holds():
    # 204 strips of 26 columns x 84 pieces of 64 rows: 17,136 work items at least
    _check(5300, 5390, [(0, 0, 90, 80), (2608, 2650, 100, 100), (5216, 5280, 84, 110), (16, 5290, 60, 100)])
