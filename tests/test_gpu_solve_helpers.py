"""Errors of the device helpers of the fixed-point kernels
(tests/solve_helpers.cu), in units of 2^-53, against extended precision."""
import os
import subprocess

import pytest

from paper_0903_4044_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_error_bounds(tmp_path):
    exe = str(tmp_path / "helpers")
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, os.path.join(HERE, "solve_helpers.cu"), "-o", exe], check=True)
    rcp, rsqrt, exp, power = map(float, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    print(rcp, rsqrt, exp, power)
    # the last operation's rounding (1); a rounding of half the weight before it for the root (e / 2), 2^-56 for the
    # exponential, ln 2 times that of log2 (1 ulp) for the power
    assert rcp <= 1.01
    assert rsqrt <= 1.6
    assert exp <= 1.2
    assert power <= 2.6
