"""NMS of small frames (at most 8,192 windows: one CTA) and the next larger ones (a cluster of
CTAs): exact against the oracle's greedy NMS on both sides of the line, with one segment of
candidates and with several."""
import os

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
W, H = 1080, 632                      # 64 x 128 = 8,192 windows


@pytest.mark.parametrize("levels", [[(W, H)], [(W, H), (64, 128)]])  # 8,192 and 8,193 windows
@pytest.mark.parametrize("n", [0, 1, 300, 2048, 2049, 8192])
@pytest.mark.parametrize("cap", [16384, 20000])                      # lists in shared and in global memory
def test_one_cta_and_cluster(levels, n, cap):
    dims = [(h // 8 - 15, w // 8 - 7) for w, h in levels]
    total = sum(r * c for r, c in dims)
    rng = np.random.default_rng(n + total)
    flat = -rng.random(total).astype(np.float32) - np.float32(0.1)
    flat[rng.permutation(total)[:n]] = rng.random(n).astype(np.float32) + np.float32(1e-3)
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    det = pd.Detector(d["w"], float(d["b"]), max_frames=1, max_width=W, max_height=H, max_candidates_per_frame=cap)
    boxes = torch.zeros(4096 * 8, dtype=torch.float32, device="cuda")
    counts = torch.full((2,), -7, dtype=torch.int32, device="cuda")
    try:
        pd.pd_nms_maps(det.h, torch.from_numpy(flat).cuda(), [r for r, _ in dims], [c for _, c in dims], levels, W, H,
                       boxes, 4096, counts)
        torch.cuda.synchronize()
        iou = float(np.float32(det.params.nms_iou))
    finally:
        det.close()
    maps, o = [], 0
    for r, c in dims:
        maps.append(flat[o:o + r * c].reshape(r, c))
        o += r * c
    ref, candidates = oracle.nms(maps, levels, W, H, threshold=0.0, iou_thr=iou, max_boxes=4096)
    kept = int(counts[0])
    assert (kept, int(counts[1])) == (len(ref), n) and candidates == n
    got = np.frombuffer(boxes.cpu().numpy().tobytes(), dtype=pd.BOX_DTYPE)[:kept]
    for f in ("level", "wx", "wy", "score", "x", "y", "w", "h"):
        assert np.array_equal(got[f], ref[f]), f
