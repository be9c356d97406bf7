"""The polynomial exponential that takes a part of the softmax off the exponential unit (csrc/umma_ptx.cuh)."""
import math
import os
import subprocess

import pytest

from paper_2508_02558_b200 import build as libbuild

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_relative_error_and_arguments_that_are_not_finite(tmp_path):
    """The polynomial's own error is 9.4e-8. Its last fused step rounds by at most 2^-24 of a value in [1, 1.42) or 2^-25 of one in
    [0.7, 1): 6.0e-8; the step before by 2^-25 of its 0.7, which reaches the result times |f| / 0.7 <= 0.71: 2.1e-8; the ones before
    that by less than 0.5e-8 together: 1.8e-7 at most. Taking the integer off and scaling by the power of two are exact. ex2.approx,
    the other exponential of the same rows, is within 2^-22."""
    exe = str(tmp_path / "poly_exp2")
    subprocess.run([libbuild._nvcc(), *libbuild.NVCC_FLAGS, "-o", exe, os.path.join(ROOT, "tests", "native", "poly_exp2.cu")], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, check=True)
    errors, special = ([float(x) for x in line.split()] for line in res.stdout.splitlines())
    assert errors[0] <= 1.8e-7 and errors[1] <= 1.8e-7, errors
    assert errors[2] <= 2**-22, errors
    nan, minus_inf, far, below, one, top, nan_sum = special
    assert math.isnan(nan) or nan >= nan_sum                    # what the rows' sums are checked for
    for x in (minus_inf, far, below):                           # clamped: 2^-126
        assert 0 < x <= 1.2e-38
    assert one == pytest.approx(1, rel=1.8e-7) and top == pytest.approx(256, rel=1.8e-7)
