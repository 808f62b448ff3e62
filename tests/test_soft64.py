"""The integer-pipe FP64 arithmetic (csrc/mcv_soft64.cuh), compiled as plain C++: division and
square root and the tests and conversions against the FPU bit for bit, with the reciprocal seeds off by up to two units
more than the hardware's; exp, log, tan and sin/cos against long double.  Bars: the
functions round one fixed-point value once (half a unit) whose own error is at most 2^-61 of
1 (sin, cos), 2^-58 of a logarithm above 0.34 (0.1 units), and for exp the error of the
reduced argument, |x| 2^-62 (0.3 units at 700)."""
import json
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1504_02776_gb300", "csrc")


def test_soft64_arithmetic(tmp_path):
    exe = str(tmp_path / "soft64_check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-I" + CSRC, "-x", "c++",
                    os.path.join(HERE, "soft64_check.cpp"), "-o", exe], check=True)
    got = json.loads(subprocess.run([exe, "400000"], check=True, capture_output=True,
                                    text=True).stdout)
    assert got["div_bad"] == 0 and got["sqrt_bad"] == 0 and got["conv_bad"] == 0, got
    assert got["exp0"] == 1.0 and got["log1"] == 0.0
    assert got["log"] <= 0.65 and got["exp"] <= 0.85 and got["tan"] <= 0.51, got
    assert got["sincos"] <= 2.0 ** -60, got
