"""Host model of the tensor-core product's arithmetic (no GPU): eight 8-bit digits
per operand, the 36 digit products with p + q <= 9 summed by diagonal, the eight
diagonal sums recombined in a 64-bit fixed-point integer with
63 - ceil(log2 n) fraction bits (at most 62) for n summed products.

Rebuilt with integers and single-precision roundings where the kernel has
them (csrc/gemm_tc.cu: put_digits, diag_fixed), and checked against rationals:
the digits give the value rounded to 62 fraction bits, ties to even; every
diagonal's sum, every value that the kernel turns into an integer by adding
1.5 2^23, and the result stay in range; the recombination is off by at most half
a unit (and the single-precision tail) from the kept digit products."""

import math
from fractions import Fraction

import numpy as np
import pytest

DIG, FRAC, KC1, KC2, LSB1, LSB2 = 8, 62, 64, 128, 57, 56


def digits(x, e):
    """Digits of x 2^(FRAC - e) rounded to an integer: its bytes with 128 added at
    every byte, minus 128 each."""
    X = round(Fraction(float(x)) * Fraction(2) ** (FRAC - e))   # ties to even
    t = (X + 0x8080808080808080) % 2 ** 64
    d = [(t >> 8 * (7 - p) & 255) - 128 for p in range(DIG)]
    assert sum(v * 2 ** (8 * (7 - p)) for p, v in enumerate(d)) == X
    return d


def whole(v):
    """The integer that v + 1.5 2^23 holds in its low mantissa bits."""
    assert abs(v) < 2 ** 22
    return round(v)


def f32(v):
    return Fraction(float(np.float32(float(v))))


def recombine(S, kc, sh):
    """diag_fixed: the sums S[0..7] of the diagonals 2..9 in units of
    2^(sh - 57) (kc 64) or 2^(sh - 56) (kc 128)."""
    x = [Fraction(v) for v in S]
    unit = Fraction(1, 8 if kc == KC1 else 16) / Fraction(2) ** sh
    if kc == KC1:
        h7 = whole(x[5] / 2)
        z = f32((x[5] - 2 * h7) * 256 + f32(x[7] / 256 + x[6]))
        P, Q, H = whole(x[4]) * 128 + h7, whole(x[2]) * 256 + whole(x[3]), whole(x[0]) * 256 + whole(x[1])
        terms = [(P, 6 - sh), (Q, 21 - sh), (H, 37 - sh)]
    else:
        h5 = whole(x[3] / 2)
        y6 = f32((x[3] - 2 * h5) * 256 + x[4])
        h6 = whole(y6 / 4)
        y7 = f32((y6 - 4 * h6) * 256 + x[5])
        h7 = whole(y7 / 4)
        z = f32((y7 - 4 * h7) * 256 + f32(x[7] / 256 + x[6]))
        P, Q, H = h6 * 256 + h7, whole(x[2]) * 128 + h5, whole(x[0]) * 256 + whole(x[1])
        terms = [(P, 6 - sh), (Q, 21 - sh), (H, 36 - sh)]
    assert all(abs(v) < 2 ** 31 for v, _ in terms) and all(s >= 0 for _, s in terms)
    return whole(z * unit) + sum(v << s for v, s in terms)


def product(a, b, general=False):
    """One real output of the sums of a[k] b[k]: (value, scale 2^(e + f), lsb)."""
    n = len(a)
    e, f = (math.frexp(float(np.abs(v).max()))[1] if np.any(v) else 0 for v in (a, b))
    ksum = -(-n // 16) * 16
    kc = KC1 if ksum <= KC1 and not general else KC2
    lsb = min(62, 63 - math.ceil(math.log2(n)))
    base = LSB1 if kc == KC1 else LSB2
    sh = min(base - lsb, 6)
    sh2 = base - lsb - sh
    da, db = [digits(v, e) for v in a], [digits(v, f) for v in b]
    R = 0
    for c0 in range(0, n, kc):
        S = [0] * 8
        for k in range(c0, min(n, c0 + kc)):
            for p in range(DIG):
                for q in range(DIG - p):
                    S[p + q] += da[k][p] * db[k][q]
        assert all(abs(v) <= 2 ** 24 for v in S)
        w = recombine(S, kc, sh)
        kept = sum(Fraction(S[d]) * Fraction(2) ** (4 - 8 * (d + 2)) for d in range(8))
        assert abs(Fraction(w) * Fraction(2) ** (sh - base) - kept) <= Fraction(2) ** (sh - base) * Fraction(17, 32)
        if sh2:
            w = round(Fraction(w, 2 ** sh2))
        R += w
    assert abs(R) < 2 ** 63
    return float(Fraction(R) * Fraction(2) ** (e + f - lsb)), 2.0 ** (e + f), lsb


def check(a, b, general=False):
    got, scale, lsb = product(a, b, general)
    exact = sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b))
    n = len(a)
    lim = (n * 2.0 ** -58.9 + -(-n // 128) * 2.0 ** -lsb) * scale + 2.0 ** -52 * abs(float(exact))
    assert abs(float(Fraction(got) - exact)) <= lim


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("n", [1, 2, 3, 7, 16, 17, 33, 64, 65, 128, 129, 300, 9000])
def test_random_products(n, general):
    rng = np.random.default_rng(n)
    for _ in range(1 if n > 1000 else 6):
        a, b = rng.standard_normal(n), rng.standard_normal(n)
        a[rng.random(n) < 0.2] *= 1e-13
        check(a, b, general)


@pytest.mark.parametrize("n", [1, 16, 64, 128])
def test_largest_digits(n):
    """All digits 64, -128 ..: every diagonal's sum at its bound."""
    v = (64 * 2 ** 56 - 128 * sum(2 ** (8 * j) for j in range(1, 7))) / 2.0 ** 62
    for s in (1.0, -1.0):
        check(np.full(n, v), np.full(n, s * v))
        check(np.full(n, 1.0 - 2.0 ** -53), np.full(n, s * (1.0 - 2.0 ** -53)))


@pytest.mark.parametrize("below", [0, 9, 10, 11, 30, 42, 43, 50, 61])
def test_entries_round_to_the_nearest_even(below):
    rng = np.random.default_rng(below)
    for x in np.ldexp(1.0 + rng.random(50), -below - 1):
        X = sum(v * 2 ** (8 * (7 - p)) for p, v in enumerate(digits(x, 0)))
        assert abs(Fraction(X) - Fraction(float(x)) * 2 ** 62) <= Fraction(1, 2)


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("n", [4, 8, 16, 17, 32, 64])
def test_one_unit_survives(n, general):
    lsb = min(62, 63 - math.ceil(math.log2(n)))
    a, b = np.zeros(n), np.zeros(n)
    a[0], a[2], b[1], b[2] = 0.5, 2.0 ** -30, 0.5, 2.0 ** (30 - lsb)
    assert product(a, b, general)[0] == 2.0 ** -lsb
