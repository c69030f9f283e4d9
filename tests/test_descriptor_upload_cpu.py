"""The pinned descriptor block is not rewritten while a copy out of it is still queued.

Every step copies its frame section from the block, and a plan for another batch shape is
written over the whole of it. pd_api.cu runs here on a CUDA runtime that holds all work
back until the host waits for it (tests/fake_runtime); whatever order of calls, the
kernels must read the descriptors of their own call, as they do one call at a time.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake_runtime") / "calls")
    src = [os.path.join(ROOT, "paper_1611_01642_gb300", "csrc", "pd_api.cu"),
           os.path.join(ROOT, "tests", "fake_runtime", "fake_runtime.cpp")]
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", os.path.join(CUDA, "include"), "-x", "c++", *src,
                        "-o", out, "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


def _log(program, calls):
    r = subprocess.run([program, *calls], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.splitlines()


@pytest.mark.parametrize("calls", ["AABA", "ABAB", "BBBAAB", "AAC", "AACA", "BBCBBA"])
def test_kernels_read_the_descriptors_of_their_own_call(program, calls):
    alone = {c: _log(program, c) for c in set(calls)}
    assert all(alone.values())
    assert _log(program, calls) == [line for c in calls for line in alone[c]]


def test_the_plan_holds_the_largest_frames_windows(program):
    """The NMS launch form follows from it; it comes with the plan, not from a walk over the levels per call."""
    pd = pytest.importorskip("paper_1611_01642_gb300")

    def windows(w, h):
        return sum(max(b // 8 - 15, 0) * max(a // 8 - 7, 0) for a, b in pd.pd_pyramid(w, h, 1.05))

    want = {"A": windows(320, 240), "B": max(windows(200, 180), windows(160, 150))}
    calls = "ABBAA"
    r = subprocess.run([program, *calls], capture_output=True, text=True, timeout=60)
    assert r.stderr.split() == [x for c in calls for x in ("windows", str(want[c]))]
