"""Performance cases of the detector: what a program that uses this framework has it do.

Whole detections (one small frame up to a mixed batch of 64), the pipelines and
options that callers select (per-block HOG, HOG-only, LBP-only, the FP32 score
kernel, upsampled levels, the learned proposal), one training step of the
proposal network, and the single stages through their own entry points.

Frames are smoothed noise with pedestrian silhouettes, the recipe of this
repository's synthetic scenes, drawn on the GPU from the seed; the SVM template
is the one that the tests and the benchmark use, the proposal parameters are the
committed checkpoint (inference) or the trainer's own initial draw (training).
"""
import math
import os

import numpy as np
import torch

import paper_1611_01642_gb300 as pd
from paper_1611_01642_gb300 import proposal

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FACTOR = float(np.float32(1.05))   # the fine pyramid of the benchmark's main workload
COARSE = float(np.float32(1.2))    # the coarse one of its latency workload
CLIP = float(np.float32(0.2))
BOXES = 1024                       # kept boxes per frame at most
LABEL = 0.0                        # a training window is positive iff its score is above this
POS_WEIGHT = 30.0                  # about negatives / positives of these scenes
LR = 1e-4                          # late in the trainer's cosine schedule
GRAD_PARTS = {"conv": (0, 14048), "head": (14048, 14210)}


def listed():
    return [
        # the smallest call: one camera frame on a coarse pyramid, latency counts
        dict(name="frame_320x240", kind="frame", w=320, h=240, coarse=True),
        # one frame of the paper's video size, boxes read before the next frame
        dict(name="frame_1242x375", kind="frame", w=1242, h=375, coarse=False),
        # a grabbed HD frame in page-locked host memory: the host-to-device step counts
        dict(name="host_1920x1080", kind="host", w=1920, h=1080, coarse=False),
        # a small detector on an odd size with 17 upsampled levels and a large candidate cap: NMS counts
        dict(name="upsampled_1241x373", kind="upsampled", w=1241, h=373, n=8, up=17),
        # the serving batch of the benchmark: score maps of 64 video frames stay on the device
        dict(name="batch_64x1242x375", kind="batch", w=1242, h=375, n=64, flags=0),
        # the largest: a mixed batch of three camera sizes
        dict(name="mixed_64", kind="mixed", a=32, b=16, c=16),
        # per-block HOG (the paper's Algorithm 5 as printed)
        dict(name="per_block_16x1242x375", kind="batch", w=1242, h=375, n=16, flags=pd.PD_FLAG_HOG_PER_BLOCK),
        # the learned proposal gating the sparse path
        dict(name="sparse_8x1920x1080", kind="sparse", w=1920, h=1080, n=8),
        # one training step of the proposal: forward, backward and Adam on every window of the batch
        dict(name="train_4x1280x720", kind="train", w=1280, h=720, n=4),
        # single stages on one level, as a caller that keeps the intermediates runs them
        dict(name="cells_1920x1080", kind="cells", w=1920, h=1080),
        dict(name="scores_240x135", kind="scores", cx=240, cy=135),
        dict(name="nms_1242x375", kind="nms", w=1242, h=375, frac=0.06),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "host", "upsampled", "batch", "batch", "mixed", "sparse", "train", "cells",
                       "scores", "nms"])
    if kind in ("frame", "host"):
        return dict(kind=kind, w=_log(rng, 96, 1920), h=_log(rng, 136, 1080), coarse=rng.random() < 0.4)
    if kind == "upsampled":
        return dict(kind=kind, w=rng.randint(320, 1300), h=rng.randint(200, 480), n=rng.randint(1, 8),
                    up=rng.randint(4, 17))
    if kind == "batch":
        flags = rng.choice([0, 0, 0, pd.PD_FLAG_HOG_ONLY, pd.PD_FLAG_LBP_ONLY, pd.PD_FLAG_SVM_FP32,
                            pd.PD_FLAG_HOG_PER_BLOCK])
        return dict(kind=kind, w=rng.randint(320, 1280), h=rng.randint(200, 720), n=_log(rng, 2, 64), flags=flags)
    if kind == "mixed":
        return dict(kind=kind, a=rng.randint(1, 32), b=rng.randint(1, 16), c=rng.randint(1, 16))
    if kind == "sparse":
        return dict(kind=kind, w=rng.randint(640, 1920), h=rng.randint(400, 1080), n=rng.randint(1, 8))
    if kind == "train":
        return dict(kind=kind, w=rng.randint(320, 1280), h=rng.randint(240, 720), n=rng.randint(1, 4))
    if kind == "cells":
        return dict(kind=kind, w=_log(rng, 64, 3840), h=_log(rng, 128, 2160))
    if kind == "scores":
        return dict(kind=kind, cx=_log(rng, 8, 480), cy=_log(rng, 16, 270))
    return dict(kind=kind, w=rng.randint(320, 1920), h=rng.randint(240, 1080), frac=round(rng.uniform(0.01, 0.06), 4))


# --------------------------------------------------------------------------- inputs
def _template():
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    return np.asarray(d["w"], np.float32), float(d["b"])


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7fffffffffff)
    return g


def _gauss():
    i = np.arange(-6, 7, dtype=np.float64)
    k = np.exp(-(i * i) / 8.0)
    return (k / k.sum()).tolist()


def _symmetric(n):
    i = torch.arange(-6, n + 6, device="cuda")
    i = torch.where(i < 0, -1 - i, i)
    return torch.where(i >= n, 2 * n - 1 - i, i).clamp_(0, n - 1)


def _smooth(a):
    """Separable Gaussian blur (sigma 2, radius 6, symmetric borders) of a 2-D float64 tensor."""
    k = _gauss()
    p = a[:, _symmetric(a.shape[1])]
    b = sum(k[d] * p[:, d:d + a.shape[1]] for d in range(13))
    p = b[_symmetric(a.shape[0])]
    return sum(k[d] * p[d:d + a.shape[0]] for d in range(13))


def _scene(seed, w, h):
    """One u8 frame [h][w] on the GPU: smoothed noise and about ten silhouettes of 48 px to 0.8 h."""
    g = _generator(seed)
    img = torch.round(_smooth(torch.randint(0, 256, (h, w), generator=g, device="cuda").double())).clamp_(0, 255)
    rng = np.random.default_rng([int(seed) & 0x7fffffff, w, h])
    for _ in range(int(rng.poisson(10.0))):
        s = float(rng.uniform(48.0, max(48.0, 0.8 * h)))
        x0 = float(rng.uniform(-0.125 * s, w - 0.375 * s))
        y0 = float(rng.uniform(-0.25 * s, h - 0.75 * s))
        c = 40.0 if rng.integers(0, 2) else -40.0
        xa, xb = max(0, math.floor(x0)), min(w, math.ceil(x0 + 0.5 * s) + 1)
        ya, yb = max(0, math.floor(y0)), min(h, math.ceil(y0 + s) + 1)
        if xa >= xb or ya >= yb:
            continue
        u = torch.arange(xa, xb, device="cuda", dtype=torch.float64)[None] + 0.5 - x0 - 0.25 * s
        v = torch.arange(ya, yb, device="cuda", dtype=torch.float64)[:, None] + 0.5 - y0
        head = (u / (0.07 * s)) ** 2 + ((v - 0.09 * s) / (0.09 * s)) ** 2 <= 1.0
        torso = (u.abs() <= 0.15 * s) & (v >= 0.18 * s) & (v < 0.58 * s)
        legs = (u.abs() >= 0.02 * s) & (u.abs() <= 0.13 * s) & (v >= 0.58 * s) & (v < s)
        sub = img[ya:yb, xa:xb]
        img[ya:yb, xa:xb] = torch.where(head | torso | legs, (sub + c).clamp(0, 255), sub)
    return img.to(torch.uint8)


def _sizes(case):
    k = case["kind"]
    if k == "mixed":
        return [(1242, 375)] * case["a"] + [(640, 480)] * case["b"] + [(1920, 1080)] * case["c"]
    return [(case["w"], case["h"])] * case.get("n", 1)


def _frames(case, seed):
    return [_scene(1000003 * (int(seed) + 1) + i, w, h) for i, (w, h) in enumerate(_sizes(case))]


def _factor(case):
    return COARSE if case.get("coarse") else FACTOR


def _level_sizes(w, h, factor, up=0):
    out = []
    for k in list(range(-up, 0)) + list(range(0, 96)):
        s = factor ** k
        a, b = math.floor(w / s + 1e-9), math.floor(h / s + 1e-9)
        if a < 64 or b < 128:
            if k >= 0:
                break
            continue
        out.append((a, b))
    return out[:96]


def _level_image(case, seed):
    return _scene(int(seed), case["w"], case["h"])


def _planes(case, seed):
    """Cell planes of a plausible level: HOG histograms and LBP counts (64 per cell), plane-major."""
    g = _generator(seed)
    cx, cy = case["cx"], case["cy"]
    pitch = max(48, (cx + 15) // 16 * 16)
    hog = torch.zeros(9, cy, pitch, device="cuda")
    r = torch.rand(9, cy, cx, generator=g, device="cuda")
    hog[:, :, :cx] = 900.0 * r * r * torch.rand(1, cy, cx, generator=g, device="cuda")
    # 64 pixels per cell over 59 bins; the non-uniform bin and a few edge patterns are the common ones
    u = torch.rand(64, cy, cx, generator=g, device="cuda")
    b = torch.where(u < 0.35, torch.full_like(u, 58.0), torch.floor(58.0 * ((u - 0.35) / 0.65) ** 2)).long().clamp_(0, 58)
    lbp = torch.zeros(59, cy, pitch, dtype=torch.uint8, device="cuda")
    n = torch.zeros(59, cy, cx, dtype=torch.int32, device="cuda")
    n.scatter_add_(0, b, torch.ones_like(b, dtype=torch.int32))
    lbp[:, :, :cx] = n.to(torch.uint8)
    return hog, lbp, pitch


def _maps(case, seed):
    """Score maps of a frame's levels, back to back: smooth fields whose top `frac` lies above 0."""
    dims = _level_sizes(case["w"], case["h"], FACTOR)
    g = _generator(seed)
    rows, cols, flat = [], [], []
    for a, b in dims:
        r, c = b // 8 - 15, a // 8 - 7
        r, c = (r, c) if r > 0 and c > 0 else (0, 0)
        rows.append(r)
        cols.append(c)
        if r:
            flat.append(_smooth(torch.randn(r, c, generator=g, device="cuda", dtype=torch.float64)).reshape(-1))
    v = torch.cat(flat) if flat else torch.zeros(1, device="cuda", dtype=torch.float64)
    cut = torch.sort(v, descending=True).values[min(v.numel() - 1, int(case["frac"] * v.numel()))]
    return (v - cut).float(), rows, cols, dims


# --------------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    w, b = _template()
    st = {"kind": kind}
    if kind in ("frame", "host", "upsampled", "batch", "mixed", "sparse", "train"):
        frames = _frames(case, seed)
        det = pd.Detector(w, b, pyr_factor=_factor(case), max_frames=len(frames),
                          max_width=max(f.shape[1] for f in frames), max_height=max(f.shape[0] for f in frames),
                          max_boxes_per_frame=BOXES, flags=case.get("flags", 0), upscale_levels=case.get("up", 0),
                          max_candidates_per_frame=65536 if kind == "upsampled" else 16384)
        if kind == "host":
            frames = [f.cpu().pin_memory() for f in frames]
        if kind == "sparse":
            params, meta = proposal.load_checkpoint(
                os.path.join(ROOT, "paper_1611_01642_gb300", "weights", "proposal_1920x1080.npz"))
            pd.pd_cnn_set_params(det.h, params)
            det.set_proposal(True, meta["keep_logit_threshold"], level_step=int(meta.get("level_step", 1)))
        if kind == "train":
            # labels are the scores of a detection on the plain path, as the trainer has them
            pd.pd_cnn_set_params(det.h, proposal.init_params(int(seed) % 1000))
            det.detect(frames)
            det.sync()
        st.update(det=det, frames=frames)
    elif kind == "cells":
        det = pd.Detector(w, b, max_frames=1, max_width=case["w"], max_height=case["h"])
        cx, cy = case["w"] // 8, case["h"] // 8
        pitch = (cx + 15) // 16 * 16
        st.update(det=det, level=_level_image(case, seed), hog=torch.zeros(9, cy, pitch, device="cuda"),
                  lbp=torch.zeros(59, cy, pitch, dtype=torch.uint8, device="cuda"), pitch=pitch, cx=cx, cy=cy)
    elif kind == "scores":
        cx, cy = case["cx"], case["cy"]
        det = pd.Detector(w, b, max_frames=1, max_width=8 * cx, max_height=8 * cy)
        hog, lbp, pitch = _planes(case, seed)
        st.update(det=det, hog=hog, lbp=lbp, pitch=pitch, cx=cx, cy=cy,
                  scores=torch.zeros(max(cy - 15, 0), max(cx - 7, 0), device="cuda"))
    else:
        det = pd.Detector(w, b, max_frames=1, max_width=case["w"], max_height=case["h"])
        maps, rows, cols, dims = _maps(case, seed)
        st.update(det=det, maps=maps, rows=rows, cols=cols, dims=dims, w=case["w"], h=case["h"],
                  boxes=torch.zeros(4096, 8, device="cuda"), counts=torch.zeros(2, dtype=torch.int32, device="cuda"))
    return st


# --------------------------------------------------------------------------- run
class _Device:
    """Device floats owned by a detector, for torch (a tensor made from it keeps the detector alive)."""

    def __init__(self, det, ptr, n):
        self.det = det
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<f4", "data": (ptr, False), "version": 3,
                                         "strides": None}


def _scores(det):
    ptr, n = pd.pd_scores(det.h)
    return torch.as_tensor(_Device(det, ptr, n), device="cuda") if n else torch.zeros(0, device="cuda")


def _boxes(det, n):
    words = np.zeros((n, BOXES, 8), np.int32)   # a frame's kept boxes, then zeros
    kept = np.zeros(n, np.int32)
    for f in range(n):
        b = det.boxes(f)
        kept[f] = len(b)
        words[f, :len(b)] = b.view(np.int32).reshape(-1, 8)
    return {"box": words[:, :, :5].view(np.float32), "window": words[:, :, 5:], "kept": kept}


def run(state):
    det, kind = state["det"], state["kind"]
    if kind == "cells":
        plane = state["cy"] * state["pitch"]
        pd.pd_cell_features(det.h, state["level"], state["hog"], plane, state["lbp"], plane, state["pitch"])
        return {"hog": state["hog"], "lbp": state["lbp"]}
    if kind == "scores":
        plane = state["cy"] * state["pitch"]
        pd.pd_window_scores(det.h, state["hog"], plane, state["lbp"], plane, state["pitch"], state["cx"], state["cy"],
                            state["scores"])
        return {"scores": state["scores"]}
    if kind == "nms":
        pd.pd_nms_maps(det.h, state["maps"], state["rows"], state["cols"], state["dims"], state["w"], state["h"],
                       state["boxes"], 4096, state["counts"])
        return {"box": state["boxes"][:, :5], "window": state["boxes"].view(torch.int32)[:, 5:],
                "counts": state["counts"]}
    if kind == "train":
        pd.pd_cnn_train_step(det.h, POS_WEIGHT, LABEL, LR)
        loss = pd.pd_cnn_train_loss(det.h)
        params, grad = pd.pd_cnn_get_params(det.h)
        return {"loss": loss, "params": params, "grad": {k: grad[a:b] for k, (a, b) in GRAD_PARTS.items()}}
    if kind == "host":
        det.detect_host(state["frames"])
    else:
        det.detect(state["frames"])
    if kind in ("batch", "mixed", "sparse"):
        return {"scores": _scores(det)}       # a device-side consumer: nothing is read back
    det.sync()
    return {"scores": _scores(det), "boxes": _boxes(det, len(state["frames"]))}


# --------------------------------------------------------------------------- work
def _windows(dims):
    return sum(max(b // 8 - 15, 0) * max(a // 8 - 7, 0) for a, b in dims)


def work(case):
    kind = case["kind"]
    if kind == "cells":
        px = case["w"] * case["h"]
        return {"bytes": px + 95 * (case["w"] // 8) * (case["h"] // 8), "flops": 55 * px}
    if kind == "scores":
        n = max(case["cx"] - 7, 0) * max(case["cy"] - 15, 0)
        return {"bytes": 95 * case["cx"] * case["cy"] + 4 * n, "flops": 19950 * n}
    if kind == "nms":
        n = _windows(_level_sizes(case["w"], case["h"], FACTOR))
        return {"bytes": 4 * n + 32 * 100, "flops": 2 * n}
    frame = px = win = 0
    for w, h in _sizes(case):
        dims = _level_sizes(w, h, _factor(case), case.get("up", 0))
        frame += w * h
        px += sum(a * b for a, b in dims)
        win += _windows(dims)
    if kind == "train":
        # the levels and the labels are read; forward, data and weight gradients of 468 MAC per pixel
        return {"bytes": px + 4 * win + 5 * 4 * 14210, "flops": 3 * 2 * 468 * px + 3 * 2 * 128 * win}
    return {"bytes": frame + 4 * win, "flops": 55 * px + 19950 * win}


# --------------------------------------------------------------------------- 64-bit values
def _q11(m, n):
    """Q11 source index and weight of m destinations over n sources (integers, rounded half up)."""
    x = torch.arange(m, device="cuda", dtype=torch.int64)
    num = ((2 * x + 1) * n - m) * 2048 + m
    q = torch.div(num, 2 * m, rounding_mode="floor")
    idx, a = q >> 11, q & 2047
    neg, end = q < 0, idx >= n - 1
    idx = torch.where(neg, torch.zeros_like(idx), torch.where(end, torch.full_like(idx, n - 1), idx))
    return idx, torch.where(neg | end, torch.zeros_like(a), a)


def _resize(f, wk, hk):
    """[B][H][W] int32 -> [B][hk][wk] int32."""
    ix, ax = _q11(wk, f.shape[2])
    iy, ay = _q11(hk, f.shape[1])
    jx, jy = (ix + 1).clamp(max=f.shape[2] - 1), (iy + 1).clamp(max=f.shape[1] - 1)
    ax, ay = ax.int(), ay.int()[:, None].long()
    t, b = f[:, iy], f[:, jy]
    top = ((2048 - ax) * t[:, :, ix] + ax * t[:, :, jx]).long()
    bot = ((2048 - ax) * b[:, :, ix] + ax * b[:, :, jx]).long()
    return (((2048 - ay) * top + ay * bot + (1 << 21)) >> 22).int()


def _edge(v, dy, dx):
    b, h, w = v.shape
    y = (torch.arange(h, device="cuda") + dy).clamp(0, h - 1)
    x = (torch.arange(w, device="cuda") + dx).clamp(0, w - 1)
    return v[:, y][:, :, x]


def _lbp_bins():
    rank, t = 0, []
    for c in range(256):
        if bin(c ^ (((c >> 1) | (c << 7)) & 255)).count("1") <= 2:
            t.append(rank)
            rank += 1
        else:
            t.append(58)
    return torch.tensor(t, device="cuda")


def _cell_index(v, hc, wc):
    """Cell number (over the batch) of every grid pixel."""
    b = v.shape[0]
    y = torch.arange(8 * hc, device="cuda") // 8
    x = torch.arange(8 * wc, device="cuda") // 8
    return ((torch.arange(b, device="cuda")[:, None, None] * hc + y[:, None]) * wc + x)


def _lbp(v):
    """[B][H][W] -> LBP cell counts [B][Hc][Wc][59] (int64)."""
    b, h, w = v.shape
    hc, wc = h // 8, w // 8
    code = torch.zeros_like(v)
    for k, (dy, dx) in enumerate([(-1, -1), (-1, 0), (-1, 1), (0, 1), (1, 1), (1, 0), (1, -1), (0, -1)]):
        code |= (_edge(v, dy, dx) >= v).int() << k
    bins = _lbp_bins()[code[:, :8 * hc, :8 * wc].long()]
    at = _cell_index(v, hc, wc) * 59 + bins
    return torch.bincount(at.reshape(-1), minlength=b * hc * wc * 59).reshape(b, hc, wc, 59)


def _votes(v):
    """Magnitude, two orientation bins and their weights of the grid pixels (float64)."""
    hc, wc = v.shape[1] // 8, v.shape[2] // 8
    gx = (_edge(v, 0, 1) - _edge(v, 0, -1))[:, :8 * hc, :8 * wc].double()
    gy = (_edge(v, 1, 0) - _edge(v, -1, 0))[:, :8 * hc, :8 * wc].double()
    th = torch.atan2(gy, gx) * (180.0 / math.pi)
    th = torch.where(th < 0, th + 180.0, th)
    th = torch.where(th >= 180.0, th - 180.0, th)
    p = th / 20.0 - 0.5
    f = torch.floor(p)
    b0 = torch.remainder(f.long(), 9)
    return torch.sqrt(gx * gx + gy * gy), (b0, torch.remainder(b0 + 1, 9)), (1.0 - (p - f), p - f)


def _hog(v):
    """[B][H][W] -> HOG cell histograms [B][Hc][Wc][9]: bilinear on one clamped grid of cells."""
    b, h, w = v.shape
    hc, wc = h // 8, w // 8
    mag, bins, wts = _votes(v)
    out = torch.zeros(b * hc * wc * 9, device="cuda", dtype=torch.float64)

    def axis(n):
        u = (torch.arange(8 * n, device="cuda", dtype=torch.float64) - 3.5) / 8.0
        f = torch.floor(u)
        return [(f.long().clamp(0, n - 1), 1.0 - (u - f)), ((f.long() + 1).clamp(0, n - 1), u - f)]

    n = torch.arange(b, device="cuda")[:, None, None]
    for cy, wy in axis(hc):
        for cx, wx in axis(wc):
            cell = (n * hc + cy[:, None]) * wc + cx
            m = mag * wy[:, None] * wx
            for q in range(2):
                out.index_add_(0, (cell * 9 + bins[q]).reshape(-1), (m * wts[q]).reshape(-1))
    return out.reshape(b, hc, wc, 9)


def _hog_blocks(v):
    """[B][H][W] -> per-block HOG [B][Hc-1][Wc-1][36]: each block binned from its own 256 pixels."""
    b, h, w = v.shape
    hc, wc = h // 8, w // 8
    mag, bins, wts = _votes(v)
    out = torch.zeros(b * (hc - 1) * (wc - 1) * 36, device="cuda", dtype=torch.float64)
    y, x = torch.arange(8 * hc, device="cuda"), torch.arange(8 * wc, device="cuda")
    n = torch.arange(b, device="cuda")[:, None, None]
    for ro in range(2):
        for co in range(2):
            by, bx = y // 8 - ro, x // 8 - co
            inside = ((by >= 0) & (by < hc - 1))[:, None] & ((bx >= 0) & (bx < wc - 1))
            block = (n * (hc - 1) + by.clamp(0, max(hc - 2, 0))[:, None]) * (wc - 1) + bx.clamp(0, max(wc - 2, 0))
            for a in range(2):
                for c in range(2):
                    wy = (1.0 - ((y - 8 * by).double() - 3.5 - 8 * a).abs() / 8.0).clamp(min=0.0)
                    wx = (1.0 - ((x - 8 * bx).double() - 3.5 - 8 * c).abs() / 8.0).clamp(min=0.0)
                    m = mag * wy[:, None] * wx * inside
                    for q in range(2):
                        at = block * 36 + 9 * (2 * a + c) + bins[q]
                        out.index_add_(0, at.reshape(-1), (m * wts[q]).reshape(-1))
    return out.reshape(b, hc - 1, wc - 1, 36)


def _score_map(hog, lbp, w, bias):
    """Score map [B][rows][cols] from cell histograms (or 36-value blocks) and LBP cell counts."""
    if hog.shape[-1] == 9:
        hog = torch.cat([hog[:, :-1, :-1], hog[:, :-1, 1:], hog[:, 1:, :-1], hog[:, 1:, 1:]], dim=3)
    f = hog / torch.sqrt((hog * hog).sum(3, keepdim=True) + 1.0)
    f = f.clamp(max=CLIP)
    f = f / torch.sqrt((f * f).sum(3, keepdim=True) + 1e-6)
    s = (lbp[:, :-1, :-1] + lbp[:, :-1, 1:] + lbp[:, 1:, :-1] + lbp[:, 1:, 1:]).double()
    s = torch.sqrt(s / s.sum(3, keepdim=True).clamp(min=1.0))
    p = torch.cat([f, s], dim=3) @ torch.from_numpy(w).cuda().double().reshape(105, 95).T  # [B][Hb][Wb][105]
    rows, cols = p.shape[1] - 14, p.shape[2] - 6
    out = torch.full((p.shape[0], rows, cols), float(bias), device="cuda", dtype=torch.float64)
    for i in range(15):
        for j in range(7):
            out += p[:, i:i + rows, j:j + cols, 7 * i + j]
    return out


def _detect64(case, seed):
    """Every frame's levels and score maps in 64 bits: [(levels [B][h][w] int32, scores [B][rows][cols])] per size."""
    w, b = _template()
    w = w.copy()
    flags = case.get("flags", 0)
    if flags & pd.PD_FLAG_HOG_ONLY:
        w[:, :, 36:] = 0.0
    if flags & pd.PD_FLAG_LBP_ONLY:
        w[:, :, :36] = 0.0
    frames, sizes = _frames(case, seed), _sizes(case)
    per_frame = [None] * len(frames)
    images = [None] * len(frames)
    for size in dict.fromkeys(sizes):
        at = [i for i, s in enumerate(sizes) if s == size]
        f = torch.stack([frames[i] for i in at]).int()
        levels, maps = [], []
        for wk, hk in _level_sizes(*size, _factor(case), case.get("up", 0)):
            v = _resize(f, wk, hk)
            levels.append(v)
            if hk // 8 > 15 and wk // 8 > 7:
                hog = _hog_blocks(v) if flags & pd.PD_FLAG_HOG_PER_BLOCK else _hog(v)
                maps.append(_score_map(hog, _lbp(v), w, b))
            else:
                maps.append(torch.zeros(len(at), 0, 0, device="cuda", dtype=torch.float64))
        for j, i in enumerate(at):
            per_frame[i] = [m[j] for m in maps]
            images[i] = [v[j] for v in levels]
    return images, per_frame


def _bf16(a):
    """Rounded to bfloat16 (ties to even), as float64."""
    m, e = torch.frexp(a)
    return torch.ldexp(torch.round(m * 256.0) / 256.0, e)


class _Stored(torch.autograd.Function):
    """An activation as it is stored (bfloat16); gradients pass."""

    @staticmethod
    def forward(ctx, a):
        return _bf16(a)

    @staticmethod
    def backward(ctx, g):
        return g


def _train64(case, seed):
    """Loss, gradient and parameters after the first Adam step, in 64 bits."""
    flat = torch.from_numpy(proposal.init_params(int(seed) % 1000)).cuda().double()
    shapes = [(16, 1, 3, 3), (16,), (32, 16, 3, 3), (32,), (32, 32, 3, 3), (32,), (32,), (1,), (16, 8), (1,)]
    ps, o = [], 0
    for s in shapes:
        n = int(np.prod(s))
        p = flat[o:o + n].reshape(s).clone()
        ps.append((_bf16(p) if len(s) == 4 else p).requires_grad_(True))
        o += n
    w1, b1, w2, b2, w3, b3, wh, bh, v, bv = ps
    images, maps = _detect64(case, seed)
    count = sum(m.numel() for f in maps for m in f)
    total = 0.0
    conv = torch.nn.functional.conv2d
    with torch.backends.cudnn.flags(enabled=False):
        for imgs, ms in zip(images, maps):
            for im, m in zip(imgs, ms):
                if not m.numel():
                    continue
                x = _bf16(im.double() / 255.0 - 0.5)[None, None]
                a1 = _Stored.apply(torch.relu(conv(x, w1, b1, stride=2, padding=1)))
                a2 = _Stored.apply(torch.relu(conv(a1, w2, b2, stride=2, padding=1)))
                a3 = torch.relu(conv(a2, w3, b3, stride=2, padding=1))
                hc, wc = im.shape[0] // 8, im.shape[1] // 8
                h = (a3[0, :, :hc, :wc] * wh[:, None, None]).sum(0) + bh
                z = conv(h[None, None], v[None, None])[0, 0] + bv
                y = (m > LABEL).double()
                sp = torch.nn.functional.softplus
                loss = (POS_WEIGHT * y * sp(-z, threshold=1000) + (1.0 - y) * sp(z, threshold=1000)).sum() / count
                loss.backward()
                total += float(loss.detach())
    grad = torch.cat([p.grad.reshape(-1) for p in ps])
    after = flat - LR * grad / (grad.abs() + 1e-8)
    return total, after, grad


def exact(case, seed):
    kind = case["kind"]
    if kind in ("nms", "sparse"):
        return None
    if kind == "cells":
        v = _level_image(case, seed).int()[None]
        cx, cy = case["w"] // 8, case["h"] // 8
        hog = torch.zeros(9, cy, (cx + 15) // 16 * 16, device="cuda", dtype=torch.float64)
        if cx and cy:
            hog[:, :, :cx] = _hog(v)[0].permute(2, 0, 1)
        return {"hog": hog, "lbp": None}
    if kind == "scores":
        w, b = _template()
        hog, lbp, _ = _planes(case, seed)
        cx = case["cx"]
        if case["cy"] < 16 or cx < 8:
            return None
        s = _score_map(hog[:, :, :cx].permute(1, 2, 0)[None].double(), lbp[:, :, :cx].permute(1, 2, 0)[None].long(), w, b)
        return {"scores": s[0]}
    if kind == "train":
        loss, after, grad = _train64(case, seed)
        return {"loss": float(loss), "params": after, "grad": {k: grad[a:b] for k, (a, b) in GRAD_PARTS.items()}}
    maps = _detect64(case, seed)[1]
    scores = torch.cat([m.reshape(-1) for f in maps for m in f])
    return {"scores": scores} if kind in ("batch", "mixed") else {"scores": scores, "boxes": None}
