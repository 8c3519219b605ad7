"""The mixed contraction's fold, step by step as the fold warps do it (packed FP32: each half rounds as
the scalar instruction does), on exact order sums of random five-digit windows:

* t = fma(o1, 2^-8, o0) and e = fma(o1, 2^-8, o0 - t) add up to o0 + o1 / 256 exactly (the orders are multiples of
  2^16 below 2^40);
* windows accumulate to within 2^-38 of sum_w 128 max|a_w| max|b_w| of the exact dot product of the
  double-float inputs.

An FP32 add or FMA here has an exact value of at most 53 bits or is rounded through exact rationals."""
import fractions
import math

import numpy as np

from test_digits_cpu import split, unnormalised_products, window_exponent

F = fractions.Fraction


def _rn(x):
    """The FP32 number nearest to the rational x (ties to even; no subnormals here)."""
    if x == 0:
        return F(0)
    e = 0
    a = abs(x)
    e = a.numerator.bit_length() - a.denominator.bit_length()
    if a < F(2) ** e:
        e -= 1
    unit = F(2) ** (e - 23)
    q = x / unit
    n = round(q)  # ties to even
    return n * unit


def _fold(o, sc, h, lo):
    """(h, lo, t, e): one window's five order sums into the running pair."""
    c8, c16 = F(1, 256), F(1, 65536)
    t = _rn(o[1] * c8 + o[0])
    e = _rn(o[1] * c8 + _rn(o[0] - t))
    tail = _rn(_rn(_rn(o[4] * c8 + o[3]) * c8 + o[2]) * c16 + e)
    p = _rn(t * sc)
    s = _rn(h + p)
    bb = _rn(s - h)
    er = _rn(_rn(h - _rn(s - bb)) + _rn(p - bb))
    l2 = _rn(lo + _rn(tail * sc + er))
    h2 = _rn(s + l2)
    return h2, _rn(l2 - _rn(h2 - s)), t, e


def test_fold_of_the_order_sums():
    rng = np.random.default_rng(9)
    worst = 0.0
    for _ in range(60):
        span = float(rng.choice([0.0, 3.0, 10.0]))
        h = lo = F(0)
        exact = bound = 0.0
        for _w in range(int(rng.integers(1, 20))):
            ah, al, a = unnormalised_products(rng, 128, span)
            bh, bl, b = unnormalised_products(rng, 128, span)
            ea, eb = window_exponent(ah), window_exponent(bh)
            da = split(ah, al, ea).astype(np.float64)
            db = split(bh, bl, eb).astype(np.float64)
            o = [F(sum(float(np.dot(da[i], db[k - i])) for i in range(k + 1))) for k in range(5)]
            assert all(_rn(x) == x and x % 65536 == 0 and abs(x) < 2 ** 40 for x in o)
            h, lo, t, e = _fold(o, F(2) ** (ea + eb - 30), h, lo)
            assert t + e == o[0] + o[1] / 256
            exact += math.fsum(a * b)
            bound += 128 * np.abs(a).max() * np.abs(b).max()
        worst = max(worst, abs(float(h + lo) - exact) / bound)
    assert worst <= 2.0 ** -38, worst


def test_fast_sum_is_exact_whichever_order_is_larger():
    rng = np.random.default_rng(10)
    for _ in range(20000):
        o0 = int(rng.integers(-2 ** 23, 2 ** 23) >> int(rng.integers(0, 24))) << 16
        o1 = int(rng.integers(-2 ** 23, 2 ** 23) >> int(rng.integers(0, 24))) << 16
        _, _, t, e = _fold([F(o0), F(o1), F(0), F(0), F(0)], F(1), F(0), F(0))
        assert t + e == F(o0) + F(o1, 256)
