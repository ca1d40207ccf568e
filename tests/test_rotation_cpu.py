"""The fixed-point rotational update (csrc/rotation.cuh) against the FP64
update it replaces, on the host: every increment it does not leave to the
FP64 code equals the FP64 one exactly, and it leaves few of them inside its
ranges (time steps, temperatures and torques of ordinary use) and all of them
outside (torques above 2^8 eps, rotations above 2^-7)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", params=["-ffp-contract=off", "-ffp-contract=fast"])
def check(request, tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("rot") / "rotation_check")
    subprocess.run(["g++", "-std=c++17", "-O2", request.param, "-I",
                    os.path.join(ROOT, "paper_1701_02059_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "csrc", "rotation_check.cpp"), "-o", exe], check=True)

    def run(*a):
        out = subprocess.run([exe, *map(str, a)], check=True, capture_output=True, text=True).stdout.split()
        return [int(x) for x in out[0::2]], [int(x) for x in out[1::2]]
    return run


@pytest.mark.parametrize("dt", [0.01, 0.001, 0.025])
@pytest.mark.parametrize("kT", [0.2, 0.01])
@pytest.mark.parametrize("torque", [2.0, 40.0])
def test_equals_fp64(check, dt, kT, torque):
    n = 200_000
    left, differ = check(dt, kT, torque, n)
    assert differ == [0, 0, 0, 0]
    # rounding-boundary cases: each part leaves well below 2 % to FP64
    assert all(x < 0.02 * n for x in left), left


def test_out_of_range_is_left_to_fp64(check):
    n = 2_000
    left, differ = check(0.01, 0.2, 1e5, n)          # torques of 10^5 eps
    assert left[0] > 0.98 * n and differ == [0, 0, 0, 0]
    left, differ = check(0.01, 2000.0, 1.0, n)       # rotations of 0.1 rad per half step
    assert left[1] > 0.98 * n and differ == [0, 0, 0, 0]
    left, differ = check(1e-9, 0.2, 1.0, n)          # a step outside the constants' range
    assert left[:3] == [n, n, n]
