"""The slicing of a transform operand's double-float value by its block's exponent, replayed in NumPy FP32
(the kernels perform the same IEEE-754 operations), over the whole range of exponents: the value is
brought to the block's scale first, so that every later step works on numbers of one size.

A value v of a block with exponent E is c_0 2^(E-8) + c_1 2^(E-16) + ... to half of the last slice's unit,
2^(E - 8 NSL - 1), for four and six slices, |c_0| <= 256 and |c_k| <= 128.  To that come the roundings of a
remainder joined in one FP32 number (NSL = 4: hi and lo after 16 bits, 2^-24 of 2^(E-17); NSL = 6: the same
after 32 bits) and, on values near the bottom of FP32's range, the lo plane's own unit of 2^-149.
"""

import numpy as np
import pytest

f = np.float32
FLOOR = -110  # the smallest block exponent (2^(16 - E) is finite down to -111)
ROUND = f(12582912.0)  # 1.5 * 2^23


def slices(hi, lo, E, nsl):
    up = np.ldexp(f(1), 16 - E).astype(f)
    rh, rl = hi * up, lo * up
    codes = []
    for k in range(0, nsl, 2):
        w = (rh + ROUND) - ROUND
        if k + 2 < nsl:
            h = rh - w
            if k + 4 < nsl:
                s = h + rl
                bb = s - h
                rh, rl = s, (h - (s - bb)) + (rl - bb)
            else:
                rh = h + rl
            rh, rl = rh * f(65536), rl * f(65536)
        c0 = (w * f(0.00390625) + ROUND) - ROUND
        codes += [c0, c0 * f(-256) + w]
    return np.array(codes, np.float64)


@pytest.mark.parametrize("nsl", [4, 6])
@pytest.mark.parametrize("E", [FLOOR, -109, -95, -91, -90, -79, -70, -40, -1, 0, 5, 60, 111])
def test_slices_carry_the_value_at_every_exponent(nsl, E):
    rng = np.random.default_rng(E + 200)
    x = rng.uniform(-1, 1, 20000) * 2.0 ** -rng.uniform(0, 40, 20000)  # of the block's largest
    x[:3] = [255.4 / 256, -255.4 / 256, 0]
    v = np.ldexp(x, E)
    hi = v.astype(f)
    lo = (v - hi.astype(np.float64)).astype(f)
    c = slices(hi, lo, E, nsl)
    assert np.all(np.abs(c[0]) <= 256) and np.all(np.abs(c[1:]) <= 128) and np.array_equal(c, np.rint(c))
    back = sum(np.ldexp(c[k], E - 8 * (k + 1)) for k in range(nsl))
    want = hi.astype(np.float64) + lo.astype(np.float64)
    last = E - 8 * nsl - 1
    joined = E - 17 - 24 if nsl == 4 else E - 33 - 24
    assert np.abs(back - want).max() <= 2.0 ** last + 2.0 ** joined


def test_smaller_blocks_take_the_floor():
    v = np.array([2.0 ** -112, 2.0 ** -120, 2.0 ** -126, -(2.0 ** -119)])
    for nsl, last in ((4, FLOOR - 33), (6, FLOOR - 49)):
        c = slices(v.astype(f), np.zeros(4, f), FLOOR, nsl)
        back = sum(np.ldexp(c[k], FLOOR - 8 * (k + 1)) for k in range(nsl))
        assert np.abs(back - v).max() <= 2.0 ** last


def test_the_kernels_floor_is_the_one_replayed():
    import os
    src = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1704_08897_gb300",
                            "csrc", "kernels_gemm_tc.cu")).read()
    assert f"return max(e, {FLOOR});" in src
