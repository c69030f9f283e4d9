"""Gradient of one training step where the training kernels' tiles can go wrong.

Their tiles are 32 x 8 and 16 x 8 positions of layers 2 and 3 (64 x 16 positions of
layer 1) and 32 x 16 windows, over all levels of all frames of a batch. The sizes
below give a single window, widths and heights one past a tile, odd sizes at every
layer, and a batch of different sizes. The reference is the oracle's network with a1
and a2 rounded to bf16 where they are stored, as the network is defined: on a single
window too few values average that rounding out. Bar per parameter tensor, as for the
other gradient test: ||gpu - ref|| <= 3e-2 ||ref||.
"""
import os

import numpy as np
import pytest

import oracle
import synth
from oracle import cnn as ocnn

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FACTOR = float(np.float32(1.3))


def _forward_stored(L, q):
    """ocnn.forward_q with a1 and a2 as they are stored (bf16)."""
    x = ocnn.input_from_level(L)
    z1 = ocnn.conv3x3_s2(x, q["w1"], q["b1"]); a1 = ocnn.bf16_round(np.maximum(z1, 0))
    z2 = ocnn.conv3x3_s2(a1, q["w2"], q["b2"]); a2 = ocnn.bf16_round(np.maximum(z2, 0))
    z3 = ocnn.conv3x3_s2(a2, q["w3"], q["b3"]); a3 = np.maximum(z3, 0)
    h = np.einsum("c,cij->ij", q["wh"], a3) + q["bh"][0]
    z = ocnn.window_pool(h, q["v"], q["bv"][0], L.shape[0] // 8 - 15, L.shape[1] // 8 - 7)
    return z, dict(q=q, x=x, z1=z1, a1=a1, z2=z2, a2=a2, z3=z3, a3=a3, h=h)


@pytest.mark.parametrize("sizes", [
    [(64, 128)],                 # one window
    [(65, 129)],                 # odd at every layer, still one window
    [(133, 137)],                # layer 2 one position past a 32-wide tile
    [(263, 141)],                # layer 3 33 wide, 2 x 18 windows
    [(317, 263)],                # several levels
    [(97, 201), (64, 128), (290, 131)],
])
def test_gradient_at_tile_edges(sizes):
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    imgs = [synth.random_image(w, h, 40 + i) for i, (w, h) in enumerate(sizes)]
    P = ocnn.init_params(5)
    for k in ("b1", "b2", "b3"):
        P[k] = P[k] + 0.05
    p32 = ocnn.flatten(P).astype(np.float32)
    det = pd.Detector(d["w"], float(d["b"]), max_frames=len(imgs), max_width=max(w for w, _ in sizes),
                      max_height=max(h for _, h in sizes), pyr_factor=FACTOR)
    try:
        pd.pd_cnn_set_params(det.h, p32)
        frames = [torch.from_numpy(im).cuda() for im in imgs]
        det.detect(frames)
        assert det.sync() == pd.PD_OK
        maps = [m.cpu().numpy() for f in range(len(imgs)) for m in det.score_maps(f)]
        levels = [oracle.resize(im, lv["width"], lv["height"]) for f, im in enumerate(imgs) for lv in det.levels(f)]
        thr = float(np.quantile(np.concatenate([m.ravel() for m in maps]), 0.9))
        pd.pd_cnn_train_step(det.h, 1.0, thr, 0.0)
        loss = pd.pd_cnn_train_loss(det.h)
        _, grad = pd.pd_cnn_get_params(det.h)
    finally:
        det.close()
    P = ocnn.unflatten(p32.astype(np.float64))
    n = sum(m.size for m in maps)
    ref_loss, ref = 0.0, {k: np.zeros(ocnn.SHAPES[k]) for k in ocnn.ORDER}
    for L, m in zip(levels, maps):
        if m.size:
            z, cache = _forward_stored(L, ocnn.rounded(P))
            part, dz = ocnn.bce_with_logits(z, (m > thr).astype(np.float64), 1.0)
            ref_loss += part * m.size / n
            for k, v in ocnn.backward(cache, dz * (m.size / n)).items():
                ref[k] += v
    assert abs(loss - ref_loss) <= 2e-2 * abs(ref_loss)
    g = ocnn.unflatten(grad.astype(np.float64))
    for k, r in ref.items():
        assert np.linalg.norm(g[k] - r) <= 3e-2 * np.linalg.norm(r) + 1e-12, k
