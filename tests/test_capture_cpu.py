"""A step's capture (csrc/capture.cuh) when one of the CUDA calls fails, on the
host with a fake of them: no failure leaves the host's notes advanced, a
capture open, a graph or a stream behind or an error pending, and the caller
learns that there is no graph.  The captured stream is the capture's own: a
caller's stream may carry other handles' work."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("cap") / "capture_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-x", "c++", "-I", os.path.join(CUDA, "include"), "-I",
                    os.path.join(ROOT, "paper_1701_02059_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "csrc", "capture_check.cpp"), "-o", exe], check=True)

    def run(fail):
        out = subprocess.run([exe, fail], check=True, capture_output=True, text=True).stdout.split()
        return dict(zip(out[0::2], map(int, out[1::2])))
    return run


@pytest.mark.parametrize("fail", ["none", "stream", "begin", "end", "end_null", "instantiate", "throw"])
def test_host_state(check, fail):
    r = check(fail)
    assert r["graph"] == (fail == "none")
    assert r["thrown"] == (fail == "throw")
    assert r["runs"] == (fail not in ("stream", "begin"))
    assert (r["note"], r["open"], r["graphs"], r["streams"], r["error"]) == (0, 0, 0, 0, 0)
    assert r["own"] == 1
