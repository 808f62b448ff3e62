"""Relative accuracy of the integer-pipe exp, log and sin/cos (csrc/mcv_soft64.cuh, compiled as
plain C++), also where the result is small: the functions they stand for are relatively accurate
everywhere, with largest measured errors of 0.53 (log), 0.89 (exp) and 1.38 units in the last
place (sin, cos).  Bar, 0.52 units: one rounding (half a unit) of a fixed-point value whose own
relative error is below 2^-60 + 2^-61, i.e. below 0.012 units where a unit is largest against the
result, and 2^-11 units of the long double reference."""
import json
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1504_02776_gb300", "csrc")


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("soft64") / "soft64_ulp_check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-I" + CSRC, "-x", "c++",
                    os.path.join(HERE, "soft64_ulp_check.cpp"), "-o", exe], check=True)
    return json.loads(subprocess.run([exe, "400000"], check=True, capture_output=True,
                                     text=True).stdout)


def test_sin_and_cos_are_relatively_accurate(errors):
    assert errors["sincos"] <= 0.52, errors


def test_exp_is_accurate_down_to_its_smallest_values(errors):
    assert errors["exp"] <= 0.52, errors


def test_log_is_accurate_next_to_one(errors):
    assert errors["log"] <= 0.52, errors
