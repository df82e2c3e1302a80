"""Arithmetic of the task graph's emulated 32 x 32 tile products (blocks above 512 rows in
the tensor-core modes), in exact integers, independent of the CUDA kernel.

With u the power of two above a row's largest entry, an entry is F u 2^-56 for an integer F,
|F| <= 2^56, written in 8 signed base-128 digits: F = sum_j d_j 2^(49 - 7 j), |d_0| <= 128,
|d_j| <= 64.  Level L = i + j of the digit products d_i e_j sums over 32 terms to |S_L| <=
2^21, exact in FP32.  Levels 0 to 5 are summed as integers in units of level 5, to which
levels 6 and 7 are rounded; the rest is dropped.  The result is off by at most 2^-48.7 u w:
2^-50 by the rounding, 7 2^17 units of level 8 (2^-70 u w each) and 1 % more by the dropped
levels, 32 (2^-57 + 2^-57) by the operands."""
from fractions import Fraction

import numpy as np
import pytest

K = 32


def _row(v):
    """(digits[k][8], u) of a row of doubles."""
    big = max(abs(x) for x in v)
    e = int(np.frexp(big)[1])                      # big < 2^e
    out = []
    for x in v:
        q = abs(Fraction(x)) * Fraction(2) ** (56 - e)
        F = (2 * q.numerator + q.denominator) // (2 * q.denominator)   # half away from zero
        F = -F if x < 0 else F
        assert abs(F) <= 2 ** 56
        hi = (F + 2 ** 27) >> 28
        d = []
        for part in (hi, F - hi * 2 ** 28):
            for sh in (21, 14, 7, 0):
                y = (part + (1 << (sh - 1))) >> sh if sh else part
                part -= y << sh
                d.append(y)
        assert sum(y * 2 ** (49 - 7 * j) for j, y in enumerate(d)) == F
        assert abs(d[0]) <= 128 and all(abs(y) <= 64 for y in d[1:])
        out.append(d)
    return np.array(out, dtype=object), Fraction(2) ** e


def _product(x, y):
    dx, u = _row(x)
    dy, w = _row(y)
    S = [sum(int(dx[k][i]) * int(dy[k][L - i]) for k in range(K) for i in range(L + 1))
         for L in range(8)]
    assert all(abs(s) <= 2 ** 21 for s in S)
    low = np.float32(float(Fraction(S[6], 2 ** 7) + Fraction(S[7], 2 ** 14)))
    tot = sum(S[L] * 2 ** (7 * (5 - L)) for L in range(6)) + int(np.rint(low))
    return Fraction(tot) * Fraction(1, 2 ** 49) * u * w, u * w


def _rows(kind, rng):
    if kind == "normal":
        return rng.standard_normal(K)
    if kind == "graded":
        return rng.standard_normal(K) * 10.0 ** rng.uniform(-12, 0, K)
    if kind == "largest":                          # every digit at its bound
        return np.where(rng.random(K) < 0.5, -1.0, 1.0) * float(2 ** 53 - 1)
    return (rng.integers(0, 2 ** 52, K) + 2 ** 52 + 0.0) * np.where(rng.random(K) < 0.5, -1, 1)


@pytest.mark.parametrize("kind", ["normal", "graded", "largest", "full"])
def test_tile_product_bound(kind):
    rng = np.random.default_rng(len(kind))
    worst = Fraction(0)
    for _ in range(24):
        x, y = _rows(kind, rng), _rows(kind, rng)
        exact = sum(Fraction(a) * Fraction(b) for a, b in zip(x, y))
        got, uw = _product(x, y)
        worst = max(worst, abs(got - exact) / uw)
    assert worst <= Fraction(2) ** -50 * Fraction(240, 100)
    assert float(2.4 * 2.0 ** -50) <= 2.0 ** -48.7


def test_levels_left_out_stay_within_their_share():
    """All digits at their bounds and of one sign: the dropped levels' largest sum."""
    d = [128] + [64] * 7
    dropped = sum(K * d[i] * d[j] * Fraction(1, 2 ** (14 + 7 * (i + j)))
                  for i in range(1, 8) for j in range(1, 8) if i + j >= 8)
    assert dropped <= Fraction(7 * 2 ** 17, 2 ** 70) * Fraction(101, 100)
