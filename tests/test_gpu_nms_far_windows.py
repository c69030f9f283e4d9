"""NMS of maps whose windows reach far beyond the frame: exact against the oracle's greedy NMS.

pd_nms_maps and pd_nms_noalloc take any map of up to 4,096 x 4,096 windows with any level
size, so a box may lie hundreds of frame widths outside the frame. Boxes there have few
float bits left: the float IoU test must leave the pairs on the threshold (3 of 5 and 1 of
3 here: neighbours 2 and 4 windows apart) to the exact one, and the culling of later
segments (threshold 0.5 and more, over 2,048 candidates) must find kept boxes there.
"""
import os

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("iou", [0.6, 1.0 / 3.0, 0.5])
@pytest.mark.parametrize("W,H,Wk,Hk,rows,cols", [
    (64, 128, 61, 128, 1, 4096),      # far to the right, one window high
    (64, 128, 64, 119, 4096, 1),      # far below
    (64, 128, 61, 119, 40, 120),      # a few widths and heights beyond, both ways
    (1000, 128, 977, 128, 1, 4096),   # from inside the frame to 33 widths beyond it
])
def test_windows_beyond_the_frame(W, H, Wk, Hk, rows, cols, iou, noalloc):
    n = rows * cols
    flat = np.random.default_rng(n + Wk).permutation(n).astype(np.float32) + np.float32(1.0)
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    boxes = torch.zeros(4096 * 8, dtype=torch.float32, device="cuda")
    counts = torch.zeros(2, dtype=torch.int32, device="cuda")
    args = (torch.from_numpy(flat).cuda(), [rows], [cols], [(Wk, Hk)], W, H)
    if noalloc:
        pd.pd_nms_noalloc(*args, 0.0, iou, 16384, boxes, 4096, counts)
        torch.cuda.synchronize()
    else:
        det = pd.Detector(d["w"], float(d["b"]), max_frames=1, max_width=W, max_height=H, nms_iou=iou)
        try:
            pd.pd_nms_maps(det.h, *args, boxes, 4096, counts)
            torch.cuda.synchronize()
        finally:
            det.close()
    ref, candidates = oracle.nms([flat.reshape(rows, cols)], [(Wk, Hk)], W, H, threshold=0.0,
                                 iou_thr=float(np.float32(iou)), max_boxes=4096)
    assert (int(counts[0]), int(counts[1])) == (len(ref), candidates) == (len(ref), n)
    got = np.frombuffer(boxes.cpu().numpy().tobytes(), dtype=pd.BOX_DTYPE)[:len(ref)]
    for f in ("level", "wx", "wy", "score", "x", "y", "w", "h"):
        assert np.array_equal(got[f], ref[f]), f
