"""The fixed-point exponential, logarithm and reciprocal of the rate kernels (csrc/fixed_math.cuh, which also
compiles for the host) against long double.

Bounds: fx_exp2 carries its result with an error below 2^-56.5 before one rounding to double, so it
is within 1/2 + 2^-56.5 2^53 = 0.59 units in the last place; fx_log2 rounds to 2^-52 once (half a
unit), on a sum whose 32-bit cubic terms add up to 2^-53.5; the conversion rounds once; the reciprocal's 62 bits
round once (half a unit and 2^-62 2^53)."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fixed") / "fixed_math_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "fixed_math_check.cpp")], check=True)
    return lambda span: [float(x) for x in subprocess.run([exe, str(span)], check=True, capture_output=True,
                                                          text=True).stdout.split()]


@pytest.mark.parametrize("span", [1.0, 30.0, 1015.0])
def test_fixed_point_functions(check, span):
    exp2_ulp, log2_units, conversion_units, rcp_ulp = check(span)
    assert exp2_ulp <= 0.59
    assert log2_units <= 0.9
    assert conversion_units <= 0.5
    assert rcp_ulp <= 0.503
