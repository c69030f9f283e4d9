"""The cells kernel inside the whole path, where a caller's cell planes do not show it.

Cell-major LBP counts: a template that is 1 at one bin of one block of the window scores
sqrt(S / 256), S that block's count of the bin (up to 256, an integer): the score is good to
2^-16 of itself (bf16 high and low part), so S comes back exactly, bin by bin. A frame of one
level; blocks from the window's first and last corner reach every cell of the level. The
reference tells every bin from its neighbours, so counts written to a wrong bin show.

Strips of up to 32 cell rows: one frame of 1242x375 is cut into strips of 2 cell rows, 16
frames into 16, 48 into 32 (a level large enough for such strips alone would have a gigabyte
of pixels). A cell row sums its votes in one order whatever the strip, so scores are the
same bits; a single frame's are compared with the oracle elsewhere.
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


def _image(W, H, seed, values):
    return (np.random.default_rng(seed).integers(0, values, size=(H, W)) * (250 // values)).astype(np.uint8)


@pytest.mark.parametrize("W,H,values,flags", [(64, 128, 3, 0), (257, 301, 2, 0), (249, 296, 4, pd.PD_FLAG_LBP_ONLY),
                                              (133, 143, 3, pd.PD_FLAG_HOG_PER_BLOCK)])
def test_cell_major_counts_are_exact(W, H, values, flags):
    img = _image(W, H, W, values)
    cells = oracle.lbp_cells(img).astype(np.int64)
    sums = cells[:-1, :-1] + cells[:-1, 1:] + cells[1:, :-1] + cells[1:, 1:]     # [blocks y][blocks x][59]
    assert all((sums[..., t] != sums[..., t + 1]).any() for t in range(58))
    rows, cols = sums.shape[0] - 14, sums.shape[1] - 6
    frame = torch.from_numpy(img).cuda()
    for i, j in [(0, 0), (14, 6), (0, 6), (14, 0)]:
        for t in range(59):
            w = np.zeros((15, 7, 95), np.float32)
            w[i, j, 36 + t] = 1.0
            det = pd.Detector(w, 0.0, pyr_factor=4.0, max_frames=1, max_width=W, max_height=H, flags=flags,
                              threshold=2.0)
            try:
                det.detect([frame])
                assert det.sync() == pd.PD_OK
                maps = det.score_maps(0)
                assert len(maps) == 1
                got = maps[0].cpu().numpy().astype(np.float64)
            finally:
                det.close()
            assert np.array_equal(np.rint(256.0 * got * got), sums[i:i + rows, j:j + cols, t]), (i, j, t)


@pytest.mark.parametrize("flags", [0, pd.PD_FLAG_HOG_PER_BLOCK, pd.PD_FLAG_HOG_PER_BLOCK | pd.PD_FLAG_HOG_ONLY,
                                   pd.PD_FLAG_HOG_ONLY, pd.PD_FLAG_LBP_ONLY])
def test_tall_strips_give_the_scores_of_short_ones(flags):
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    frames = [torch.from_numpy(synth.make_scene(1242, 375, 2, 300 + i)).cuda() for i in range(4)]
    det = pd.Detector(d["w"], float(d["b"]), max_frames=48, max_width=1242, max_height=375, flags=flags)
    try:
        def scores(batch):
            det.detect(batch)
            assert det.sync() in (pd.PD_OK, pd.PD_EOVERFLOW)
            return [torch.cat([m.reshape(-1) for m in det.score_maps(f)]).clone() for f in range(len(batch))]

        alone = [scores([f])[0] for f in frames]
        for n in (16, 48):
            got = scores([frames[i % 4] for i in range(n)])
            for i in range(n):
                assert torch.equal(got[i], alone[i % 4]), (n, i)
    finally:
        torch.cuda.synchronize()
        det.close()
