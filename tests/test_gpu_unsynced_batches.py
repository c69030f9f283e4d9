"""Batches of changing shape, one after the other without a wait: every call's scores are
those of a fresh handle, the same bits. The stream is kept busy, so the copies of a call
are still queued when the next call is planned; repeated shapes go through the captured
graph."""
import os

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _scores(det, n):
    return torch.cat([m.reshape(-1) for f in range(n) for m in det.score_maps(f)]).clone()  # stream-ordered


@pytest.mark.parametrize("calls", ["AABA", "ABBAAB"])
def test_scores_are_those_of_fresh_handles(calls):
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    batch = {"A": [synth.make_scene(320, 240, 1, 7)],
             "B": [synth.make_scene(200, 180, 1, 8), synth.make_scene(301, 233, 1, 9)]}
    batch = {k: [torch.from_numpy(f).cuda() for f in v] for k, v in batch.items()}
    make = lambda: pd.Detector(d["w"], float(d["b"]), max_frames=2, max_width=320, max_height=240)  # noqa: E731
    want = {}
    for k, frames in batch.items():
        det = make()
        try:
            det.detect(frames)
            assert det.sync() == pd.PD_OK
            want[k] = _scores(det, len(frames))
        finally:
            det.close()
    busy = torch.zeros(1 << 28, device="cuda")
    det = make()
    try:
        torch.cuda.synchronize()
        for _ in range(40):  # some 10 ms of work before the first call's copies
            busy.add_(1.0)
        got = []
        for c in calls:
            det.detect(batch[c])
            got.append(_scores(det, len(batch[c])))
        assert det.sync() == pd.PD_OK
    finally:
        det.close()
    for c, g in zip(calls, got):
        assert torch.equal(g, want[c]), c
