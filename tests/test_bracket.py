"""The root of one grid cell of the FP64 crystal kernel (csrc/mcv_bracket.cuh, compiled as plain
C++) against plain bisection: functions on which a secant iteration closes slowly (a kink, a jump,
roots of fractional order, exponential growth) and cells with three roots, one of them next to
the first midpoint.  Bars: the same root in every cell; its distance
within 2^-50 of the cell (what the bisection leaves) plus two neighbouring doubles, unless g is its
own rounding there; at most 86 evaluations (12 undecided midpoints while the bracket is wider than
2^-12 of the cell, its two ends, 60 steps, and 12 where the last steps of the bisection follow)."""
import json
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1504_02776_gb300", "csrc")


def test_bracketed_root_is_the_bisections(tmp_path):
    exe = str(tmp_path / "bracket_check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-I" + CSRC, "-x", "c++",
                    os.path.join(HERE, "bracket_check.cpp"), "-o", exe], check=True)
    got = json.loads(subprocess.run([exe, "300000"], check=True, capture_output=True,
                                    text=True).stdout)
    assert got["other"] == 0 and got["far"] <= 1.0, got
    assert got["most"] <= 86 and got["smooth"] < 8.0, got
