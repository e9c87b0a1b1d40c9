"""Integer products of binary64 weights (CPU, emulated): a weight is split into
its first 32 bits A and the next 31 bits B in units of its grid's scale, and the
pair's product is V = round(P / 2^15), P = A' A_j + 2 t, with A' the halved i-side
and t the high words of the cross products.  V must stay within one unit and the
dropped terms of the exact product, below 2^48 + 1, and its pieces (16, 16 and 17
bits; 9, 20 and 20 where the count shares the first word) must add up to it, also
over as many products as a record takes between flushes."""

import random
from fractions import Fraction

import pytest


def _split(w, emax):
    """(A, B) of a float w < 2^(emax - 126) as weight_hi, weight_lo: w 2^(158 - emax)."""
    x = Fraction(w) * Fraction(2) ** (158 - emax)
    a = int(x)
    return a, int((x - a) * 2 ** 31)


def _product(ai, bi, aj, bj):
    wb = ((ai & 1) << 30) | (bi >> 1)
    wi = ai >> 1
    t = ((wi * bj) >> 32) + ((wb * aj) >> 32) + 0x2000
    assert t < 2 ** 32
    p = t * 2 + wi * aj
    assert p < 2 ** 64
    return p >> 15


@pytest.mark.parametrize("span_i,span_j", [(0, 0), (1, 3), (4, 8), (6, 6), (8, 4)])
def test_products_of_63_bits(span_i, span_j):
    rng = random.Random(100 * span_i + span_j)
    emax = 127                                    # weights in [2^-span, 2)
    for n in range(20000):
        w = [rng.uniform(1.0, 2.0) * 2.0 ** -rng.randint(0, s) for s in (span_i, span_j)]
        if n < 4:                                 # the largest, and powers of two
            w = [[2.0 - 2.0 ** -52] * 2, [1.0, 2.0 - 2.0 ** -52], [2.0 ** -span_i, 2.0 ** -span_j], [1.0, 1.0]][n]
        (ai, bi), (aj, bj) = _split(w[0], emax), _split(w[1], emax)
        assert ai < 2 ** 32 and aj < 2 ** 32
        v = _product(ai, bi, aj, bj)
        assert 0 <= v <= 2 ** 48
        exact = Fraction(w[0]) * Fraction(w[1]) * Fraction(2) ** (2 * (158 - emax)) / 2 ** 16
        assert abs(v - exact) < Fraction(1, 2) + Fraction(8, 2 ** 15)
        assert (v & 0xFFFF) + ((v >> 16 & 0xFFFF) << 16) + ((v >> 32) << 32) == v
        assert (v & 0x1FF) + ((v >> 9 & 0xFFFFF) << 9) + ((v >> 29) << 29) == v


def test_records_do_not_wrap():
    top = 2 ** 48                                 # largest V
    for v in (top, top - 1):
        assert 2 ** 15 * (v >> 32) < 2 ** 32 and 2 ** 15 * 0xFFFF < 2 ** 32
        assert 2047 * 0x1FF < 2 ** 20 and 2047 * 0xFFFFF < 2 ** 32 and 2047 * (v >> 29) < 2 ** 32
    # binary32 weights: P >> 16 below 2^48 in pieces of 8, 20 and 20 bits
    assert 4095 * 0xFF < 2 ** 20 and 4095 * 0xFFFFF < 2 ** 32 and 4095 < 2 ** 12
    p = random.Random(1).getrandbits(64)
    lo, hi = p & 0xFFFFFFFF, p >> 32
    x, y, z = (lo >> 16) & 0xFF, ((p >> 24) & 0xFFFFFFFF) & 0xFFFFF, hi >> 12
    assert x + (y << 8) + (z << 28) == p >> 16
