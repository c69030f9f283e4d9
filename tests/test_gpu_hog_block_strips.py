"""Per-block HOG on the warp-per-strip cells kernel at the edges of its strips
(15 cells wide, 2 to 32 cell rows tall), against the oracle's blocks.

Tolerance, per histogram value: the vote angle is within 3.3e-7 bin
(polynomial) plus a few float32 roundings of a position below 9 bins (4 x
5.4e-7), the magnitude within 2^-21, and a value sums at most 12 rows and 12
columns of non-negative votes in float32 (at most 24 roundings of 6e-8 each):
under 4.5e-6 of the block's mass; 1e-5 is asserted.
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
TOL = 1e-5


# one strip and one cell more or less on each axis, 2-row strips with a remainder, strips of 32
# rows (2,400 x 1,800: enough of them for full height), rows that end off a cell edge
@pytest.mark.parametrize("W,H", [(16, 24), (112, 64), (120, 264), (128, 256), (135, 271), (249, 40), (2400, 1800)])
@pytest.mark.parametrize("shift", [0, 1])  # byte offset of the level: 1 takes the clamped byte loads
def test_blocks_at_strip_edges(W, H, shift):
    from paper_1611_01642_gb300 import build as bld
    bld.build()
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    L = synth.random_image(W, H, 31 * W + H, smooth=H > 100)
    Hc, Wc = H // 8, W // 8
    cp = ((Wc + 15) // 16) * 16
    plane = Hc * cp
    pitch = W + 3 * shift
    buf = torch.zeros((H * pitch + 16,), dtype=torch.uint8, device="cuda")
    level = buf[shift:shift + H * pitch].view(H, pitch)[:, :W]
    level.copy_(torch.from_numpy(L))
    hog = torch.full((36 * plane,), float("nan"), dtype=torch.float32, device="cuda")
    lbp = torch.full((59 * plane,), 255, dtype=torch.uint8, device="cuda")
    h = pd.Detector(d["w"], float(d["b"]), max_frames=1, max_width=max(W, 64), max_height=max(H, 128),
                    flags=pd.PD_FLAG_HOG_PER_BLOCK)
    try:
        pd.pd_cell_features(h.h, level, hog, plane, lbp, plane, cp)
        torch.cuda.synchronize()
    finally:
        h.close()
    q = hog.cpu().numpy().reshape(4, 9, Hc, cp)[..., :Wc].astype(np.float64)
    got = np.concatenate([q[0, :, :-1, :-1], q[1, :, :-1, 1:], q[2, :, 1:, :-1], q[3, :, 1:, 1:]],
                         axis=0).transpose(1, 2, 0)
    ref = oracle.hog_blocks(L)
    err = np.abs(got - ref) - TOL * ref.sum(axis=2, keepdims=True) - 1e-6
    assert np.all(err <= 0), float(err.max())
    lg = lbp.cpu().numpy().reshape(59, Hc, cp)[:, :, :Wc].transpose(1, 2, 0)
    assert np.array_equal(lg, oracle.lbp_cells(L))
