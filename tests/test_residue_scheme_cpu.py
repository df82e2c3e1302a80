"""Arithmetic of the emulated FP64 products in residues, checked on the CPU with exact
integers, independent of the CUDA kernels (modular products with recovery by the Chinese
remainder theorem, as in arXiv 2504.08009).

* Residues.  |F| <= 2^56 in four signed 14-bit digits, t = d0 + d1 c1 + d2 c2 + d3 c3 with
  the residues c of 2^14, 2^28, 2^42: |t| < 2^23, and t minus p times the FP32-rounded t / p
  is congruent to F with magnitude at most p / 2, so exact in BF16.
* Sums.  256 products of residues stay below 2^24, exact in FP32.
* Recovery.  Two residues meet in a 27-bit integer, seven such integers times 113-bit
  fractions give X / P modulo 1 within 2^40 / P; |X| <= K 2^112 is recovered up to K = 4847.
"""
import math
import random

import numpy as np
import pytest

MODULI = [511, 509, 508, 505, 503, 501, 499, 493, 491, 487, 481, 479, 473, 467]
P = math.prod(MODULI)
FRAC = 113


def _sym(a, p):
    r = a % p
    return r - p if r > p // 2 else r


def _signed14(x):
    return ((x & 0x3FFF) ^ 0x2000) - 0x2000


def _residues(F):
    hi = (F + (1 << 27)) >> 28
    lo = F - (hi << 28)
    d0, d2 = _signed14(lo), _signed14(hi)
    d1, d3 = (lo - d0) >> 14, (hi - d2) >> 14
    out = []
    for p in MODULI:
        t = d0 + sum(d * _sym(1 << (14 * i), p) for i, d in ((1, d1), (2, d2), (3, d3)))
        assert abs(t) < 1 << 23
        q = round(float(t) * float(np.float32(1) / np.float32(p)))   # one rounding, as an FMA
        out.append(t - q * p)
    return out


def _tables():
    w = [_sym(pow(P // p, -1, p), p) for p in MODULI]
    pairs, offset = [], 0
    for i in range(0, len(MODULI), 2):
        a, b = w[i] * MODULI[i + 1], w[i + 1] * MODULI[i]
        c = (-512 * a if a < 0 else 0) + (-512 * b if b < 0 else 0)
        pp = MODULI[i] * MODULI[i + 1]
        f = ((1 << FRAC) + pp // 2) // pp
        assert f < 1 << 96
        pairs.append((a, b, c, f))
        offset -= (256 * (a + b) + c) * f
    return pairs, offset % (1 << FRAC)


def _recover(r):
    """T with X = T P 2^-113, as the kernel's three 64-bit limbs form it."""
    pairs, off = _tables()
    limb = [off & 0xFFFFFFFF, off >> 32 & 0xFFFFFFFF, off >> 64]
    for i, (a, b, c, f) in enumerate(pairs):
        y = (r[2 * i + 1] + 256) * b + (r[2 * i] + 256) * a + c
        assert 0 <= y < 1 << 27
        for j in range(3):
            limb[j] += y * (f >> 32 * j & 0xFFFFFFFF)
    assert max(limb) < 1 << 64
    t = ((limb[2] << 64) + (limb[1] << 32) + limb[0]) % (1 << FRAC)
    return t - (1 << FRAC) if t >> (FRAC - 1) else t


def test_moduli():
    assert all(math.gcd(p, q) == 1 for i, p in enumerate(MODULI) for q in MODULI[:i])
    assert 1 << 125 <= P < 1 << 126
    assert 2 * 4847 << 112 <= P - (1 << 42) and 2 * 5120 << 110 <= P
    assert 256 * 255 * 255 + 255 <= 1 << 24


def test_residues_are_congruent_and_small():
    rng = random.Random(1)
    edge = [0, 1, -1, 1 << 56, -(1 << 56), (1 << 56) - 1, 1 << 55, (1 << 28) - 1, -(1 << 27)]
    for F in edge + [rng.randint(-(1 << 56), 1 << 56) for _ in range(20000)]:
        for r, p in zip(_residues(F), MODULI):
            assert (r - F) % p == 0 and abs(r) <= p // 2


@pytest.mark.parametrize("K", [1, 7, 256, 4847])
def test_products_are_recovered(K):
    rng = random.Random(K)
    for trial in range(20):
        a = [rng.randint(-(1 << 56), 1 << 56) for _ in range(K)]
        b = [rng.randint(-(1 << 56), 1 << 56) for _ in range(K)]
        if trial == 0:
            a = b = [1 << 56] * K
        X = sum(x * y for x, y in zip(a, b))
        t = _recover([_sym(X, p) for p in MODULI])
        assert abs(t * P - (X << FRAC)) <= 1 << (40 + FRAC)


def test_zero_is_exact_and_sign_symmetric():
    assert _recover([0] * len(MODULI)) == 0
    rng = random.Random(3)
    for _ in range(2000):
        X = rng.randint(1, 1 << rng.randint(1, 124))
        r = [_sym(X, p) for p in MODULI]
        assert _recover(r) == -_recover([-v for v in r])
