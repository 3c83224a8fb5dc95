"""The FP64 builds' reciprocal (rcp_newton in rb_summary.cu): the FP32 seed of
test_rcp_newton and one third-order step r + r (e + e^2), e = 1 - S r, emulated
with exactly rounded fused multiply-adds.  The step's truncation is e^3 < 2^-66, its
roundings half an ulp of r and 2^-75, so the result is within 1 ulp of 1/S."""
import math
from fractions import Fraction

import numpy as np
import pytest

from tests.test_rcp_newton import _fma, _rcp_newton


@pytest.mark.parametrize("lo,hi,n", [(-49, -38, 2000), (-307, 306, 1000), (-1, 1, 1000)])
def test_third_order_step_within_one_ulp(lo, hi, n):
    rng = np.random.default_rng(7)
    values = list(10.0 ** rng.uniform(lo, hi, n)) + [1.0, 2.0, 3.0, float(np.nextafter(2.0, 0.0)), float(np.nextafter(1.0, 2.0)),
                                                     2.0 ** -1022, 2.0 ** 1020, float(np.nextafter(2.0 ** 1021, 0.0))]
    for S in map(float, values):
        r0, _ = _rcp_newton(S)  # the seed (or the division, outside the routine's range)
        e = _fma(-S, r0, 1.0)
        r = _fma(r0, _fma(e, e, e), r0)
        exact = Fraction(1) / Fraction(S)
        assert abs(e) < 2.0 ** -22 and float(abs(Fraction(r) - exact)) <= math.ulp(float(exact)), S
