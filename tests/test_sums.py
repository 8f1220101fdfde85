"""Sums across lanes and warps that stand for FP64 ones: the three-number FP32 sum (Sum3) replayed in NumPy
(the kernels perform the same IEEE-754 operations), and which sums use it.

The bound of its FP64 value against the exact sum, relative to the sum of magnitudes: the additions to the
third number are the only roundings, of numbers below 2^-46 of the total (n additions of numbers 2^-24
below a number 2^-24 below the total, n <= 2^10), so below 2^-60 in all; the two additions of its value in
FP64 round by 2^-53 each: 2^-51.  FP64 butterflies over the same ten levels round by 10 2^-53 at worst."""

import os
import re
from fractions import Fraction

import numpy as np
import pytest

f = np.float32
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1704_08897_gb300", "csrc")


def two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def join(x, y):
    s, e = two_sum(x[0], y[0])
    c, t = two_sum(x[1], y[1])
    d = x[2] + (y[2] + t)
    c, t = two_sum(c, e)
    return s, c, d + t


def butterfly(x, width):
    n = width
    while n > 1:
        n //= 2
        x = join(tuple(v[..., :n] for v in x), tuple(v[..., n:2 * n] for v in x))
    return tuple(v[..., 0] for v in x)


@pytest.mark.parametrize("warps", [4, 8, 16])
@pytest.mark.parametrize("spread", [0, 3, 8])
def test_three_numbers_carry_a_sum_as_fp64_does(warps, spread):
    rng = np.random.default_rng(warps + spread)
    for _ in range(20):
        s = (rng.standard_normal((warps, 32)) * 10.0 ** rng.uniform(-spread, 0, (warps, 32))).astype(f)
        c = (s * rng.uniform(-2.0 ** -23, 2.0 ** -23, s.shape)).astype(f)
        exact = sum(Fraction(float(v)) for v in np.concatenate([s.ravel(), c.ravel()]))
        size = sum(abs(Fraction(float(v))) for v in s.ravel())
        x = butterfly(butterfly((s, c, np.zeros_like(s)), 32), warps)
        value = float(x[0]) + (float(x[1]) + float(x[2]))
        assert abs(Fraction(value) - exact) <= size / 2 ** 51


def test_the_preconditioners_and_the_3d_sums_use_them():
    def code(name):
        return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    tc, box = code("kernels_gemm_tc.cu"), code("solve3d.cu")
    assert "group_sum_pair" not in tc and "group_sum_pair" not in box and "block_sum_comp" not in box
    # r.z and z.q of stage 3 and of the unfold, in FP32 mode; r.r and r.z of a box
    assert len(re.findall(r"reduce_dots<32, DOTS3>\(\w+\)", tc)) == 4
    assert code("api.cu").count("dots3 = ctx->opt.prec == EXT_PREC_FP32;") == 2
    assert len(re.findall(r"\.reduce<32>\(\)", box)) == 2
