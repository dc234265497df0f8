"""Error bounds of the fixed-point arithmetic of the FP64 step, on the host
(tests/fixed_arithmetic.cpp): results rounded once to 53 bits carry half an
ulp (2^-53 of the value) and the truncations of their 60-bit intermediates."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_error_bounds(tmp_path):
    exe = str(tmp_path / "fixed")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(HERE, "..", "paper_0903_4044_gb300", "csrc"), "-x",
                    "c++", os.path.join(HERE, "fixed_arithmetic.cpp"), "-o", exe], check=True)
    combine, units96, gauss, relax, wide, add96, fix58 = map(float, subprocess.run([exe], check=True, capture_output=True,
                                                                   text=True).stdout.split())
    half = 2.0 ** -53
    assert combine <= half + 2.0 ** -54   # the sum keeps at least 54 bits above three truncations of 2^-60
    assert gauss <= half + 2.0 ** -56 + 6 * 2.0 ** -58  # 2^-56.6 of the series, 2 w dw ln 2 of the argument (w < 8, dw 2^-59)
    assert relax <= half + 2.0 ** -55
    assert wide <= half + 2.0 ** -60
    assert units96 == 0.0  # truncated
    assert add96 <= 0.5  # rounded
    assert fix58 <= 0.5
