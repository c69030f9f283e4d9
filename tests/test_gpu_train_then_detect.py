"""A sparse detection right after a training step that is still running on another stream uses the
trained parameters: its logits are, bit for bit, those of a fresh handle loaded with them."""
import os

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_1611_01642_gb300")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_detect_waits_for_training_on_another_stream():
    from paper_1611_01642_gb300 import proposal
    d = np.load(os.path.join(ROOT, "tests", "golden", "svm_template_seed0.npz"))
    frame = torch.from_numpy(synth.make_scene(320, 240, 2, 21)).cuda()
    busy = torch.zeros(1 << 28, device="cuda")
    make = lambda: pd.Detector(d["w"], float(d["b"]), max_frames=1, max_width=320, max_height=240)  # noqa: E731
    logits = lambda det: torch.cat([m.reshape(-1) for m in det.logit_maps(0)]).clone()  # noqa: E731
    det, first = make(), proposal.init_params(3)
    train, other = torch.cuda.Stream(), torch.cuda.Stream()
    try:
        pd.pd_cnn_set_params(det.h, first)
        det.detect([frame])
        det.sync()
        torch.cuda.synchronize()
        with torch.cuda.stream(train):
            for _ in range(20):
                busy.add_(1.0)
            pd.pd_cnn_train_step(det.h, 30.0, 0.0, 1e-2)
        with torch.cuda.stream(other):
            det.set_proposal(True, 0.0)
            det.detect([frame])
            assert det.sync() in (pd.PD_OK, pd.PD_EOVERFLOW)
            got = logits(det)
        torch.cuda.synchronize()
        params = pd.pd_cnn_get_params(det.h)[0]
    finally:
        det.close()
    assert not np.array_equal(params, first)
    fresh = make()
    try:
        pd.pd_cnn_set_params(fresh.h, params)
        fresh.set_proposal(True, 0.0)
        fresh.detect([frame])
        assert fresh.sync() in (pd.PD_OK, pd.PD_EOVERFLOW)
        assert torch.equal(logits(fresh), got)
        torch.cuda.synchronize()
    finally:
        fresh.close()
