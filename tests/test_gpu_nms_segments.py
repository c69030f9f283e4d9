"""NMS where its segments, lists and sorts can go wrong: exact against the oracle's greedy NMS.

The best 2,048 candidates are sorted and walked at a time, up to 256 of them by counting,
more by the score's place in its range or, where scores hardly differ, by a bitonic
network; the rest waits in lists (global memory with a cap above 16,384). Candidate counts
lie at the edges of these, scores are spread, tied (few values), all equal, or one far
above the rest; the threshold is 0.5 (culling applies), 0.3 (it does not) and 0.
"""
import os

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
W, H = 1242, 375
LEVELS = oracle.pyramid(W, H, float(np.float32(1.05)))
DIMS = [(h // 8 - 15, w // 8 - 7) for w, h in LEVELS]


def _maps(n, kind, seed):
    rng = np.random.default_rng(seed)
    total = sum(r * c for r, c in DIMS)
    flat = -rng.random(total).astype(np.float32) - np.float32(0.1)
    at = rng.permutation(total)[:n]
    v = {"spread": lambda: rng.random(n) + 1e-3, "tied": lambda: rng.integers(1, 9, n) * 0.25,
         "equal": lambda: np.full(n, 0.75), "outlier": lambda: np.where(np.arange(n) == 0, 1e6, rng.random(n) + 1e-3)}
    flat[at] = v[kind]().astype(np.float32)
    return flat


@pytest.mark.parametrize("n,kind,iou,cap,max_boxes", [
    (1, "spread", 0.5, 16384, 4096), (256, "tied", 0.5, 16384, 4096), (257, "spread", 0.5, 16384, 4096),
    (1025, "equal", 0.5, 16384, 4096), (2048, "spread", 0.3, 16384, 4096), (2049, "spread", 0.5, 16384, 4096),
    (5000, "tied", 0.5, 16384, 4096), (5000, "equal", 0.3, 16384, 4096), (9000, "outlier", 0.5, 16384, 300),
    (16384, "spread", 0.5, 16384, 4096), (3000, "spread", 0.0, 16384, 4096), (2049, "tied", 0.5, 20000, 4096),
    (18000, "spread", 0.5, 65536, 4096),
])
def test_segments_match_the_sequential_walk(n, kind, iou, cap, max_boxes):
    flat = _maps(n, kind, n + len(kind))
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    det = pd.Detector(d["w"], float(d["b"]), max_frames=1, max_width=W, max_height=H, nms_iou=iou,
                      max_candidates_per_frame=cap, max_boxes_per_frame=max_boxes)
    rows, cols = [r for r, _ in DIMS], [c for _, c in DIMS]
    boxes = torch.zeros(max_boxes * 8, dtype=torch.float32, device="cuda")
    counts = torch.zeros(2, dtype=torch.int32, device="cuda")
    try:
        pd.pd_nms_maps(det.h, torch.from_numpy(flat).cuda(), rows, cols, LEVELS, W, H, boxes, max_boxes, counts)
        torch.cuda.synchronize()
    finally:
        det.close()
    maps, o = [], 0
    for r, c in DIMS:
        maps.append(flat[o:o + r * c].reshape(r, c))
        o += r * c
    ref, candidates = oracle.nms(maps, LEVELS, W, H, threshold=0.0, iou_thr=float(np.float32(iou)), max_boxes=max_boxes)
    kept = int(counts[0])
    assert (kept, int(counts[1])) == (len(ref), candidates) == (len(ref), n)
    got = np.frombuffer(boxes.cpu().numpy().tobytes(), dtype=pd.BOX_DTYPE)[:kept]
    for f in ("level", "wx", "wy", "score", "x", "y", "w", "h"):
        assert np.array_equal(got[f], ref[f]), f
