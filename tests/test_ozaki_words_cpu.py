"""The word arithmetic of the Ozaki kernels, emulated bit by bit with Python integers, no device needed:

* oz_frac_value (csrc/gemm_oz.cu): carries of the eleven byte sums, one's-complement magnitude, normalisation, the product
  with the leading 64 bits of P, rounding.  The value lies within 2^-77 P + 2^-52.9 |x| of the integer x, its sign is
  x's, a value past the snapping threshold is kept and one below 2^11 units of 2^-88 P is a zero;
* the base-256 digits of the O(r^5) products (csrc/acse_zoz.cu): X = round(x 2^(8D + 1 - e)) through one FMA with
  1.5 2^52 + bias, its bytes as digits (the leading one within -256 .. 256, the others -128 .. 127), level sums exact in
  FP32 and within the integer ranges of the epilogue, and the assembled product within the fixed-point rounding of
  both rows."""
import math
import random
from fractions import Fraction

import pytest

from tests.test_ozaki_fraction_cpu import FL, _value

M32, M64 = 2 ** 32 - 1, 2 ** 64 - 1


def _s32(v):
    v &= M32
    return v - 2 ** 32 if v >> 31 else v


def _frac_value(a, Pm, ex):
    """(significand of 53 bits with sign, exponent) as oz_frac_value forms them, or (0, 0)."""
    assert len(a) == FL and all(abs(v) < 2 ** 21 for v in a)
    t0 = a[0] * 256 + (a[1] + a[2] * 256) * 65536
    t1 = a[3] + a[4] * 256 + (a[5] + a[6] * 256) * 65536
    t2 = a[7] + a[8] * 256 + (a[9] + a[10] * 256) * 65536
    u1 = t1 + (t0 >> 32)
    u2 = t2 + (u1 >> 32)
    sg = M32 if _s32(u2) < 0 else 0
    w0, w1, w2 = (t0 & M32) ^ sg, (u1 & M32) ^ sg, (u2 & M32) ^ sg
    if w2 == 0:
        if w1 == 0 and w0 < 1 << 19:
            return 0, 0
        w2, w1, w0, ex = w1, w0, 0, ex - 32
        if w2 == 0:
            w2, w1, ex = w1, 0, ex - 32
    n = 32 - w2.bit_length()
    top = (((w2 << 64 | w1 << 32 | w0) << n) >> 32) & M64
    assert top >> 63
    m = (top * Pm) >> 64
    assert 2 ** 62 <= m < 2 ** 64
    e = ex - n
    s = (m >> 63) ^ 1
    m <<= s
    e -= s
    q = (m >> 11) + ((m >> 10) & 1)
    return (-q if sg else q), e + 11


@pytest.mark.parametrize("nch", [1, 2])
@pytest.mark.parametrize("T", [9, 13, 16, 17, 19])
def test_fraction_words(T, nch):
    rng = random.Random(7 * T + nch)
    P = _value(0, T, nch, rng)[3]
    Pe = P.bit_length() - 64
    Pm = P >> Pe if Pe >= 0 else P << -Pe
    unit = Fraction(P, 2 ** 88)
    edge = [int(unit * k) * s for s in (1, -1) for k in (2 ** 12 + 2 ** 11, 2 ** 20, 2 ** 24 - 1, 2 ** 24, 2 ** 56 - 1, 2 ** 56, 2 ** 56 + 1)]
    xs = [0, P // 4, -(P // 4)] + [x for x in edge if abs(x) <= P // 4]
    xs += [rng.choice((-1, 1)) * (rng.randrange(P // 4 + 1) >> rng.randrange(0, 100)) for _ in range(400)]
    for x in xs:
        F, ws, sums, _ = _value(x, T, nch, rng)
        q, e = _frac_value(sums, Pm, Pe)
        v = Fraction(q) * Fraction(2) ** e
        assert abs(v - x) <= unit * 2 ** 11 * 2 + Fraction(abs(x)) * Fraction(2) ** -53 * Fraction(1 + 2.0 ** -4), (x, v)
        if x == 0:
            assert q == 0
        elif abs(x) >= unit * 2 ** 12:                # past the threshold by more than the constants' error: kept
            assert q != 0 and (q > 0) == (x > 0) and 2 ** 52 <= abs(q) <= 2 ** 53


def _row_exp(row):
    """e of rz_row_exp from the upper words of the row."""
    import struct

    hi = max((struct.unpack("<Q", struct.pack("<d", v))[0] >> 32) & 0x7FFFFFFF for v in row)
    return 0 if hi == 0 else min(1000, max(-960, (hi >> 20) - 1023 + 2))


def _digits(x, e, D):
    """D digits, most significant first, of X, and X."""
    bias = sum(128 << (8 * i) for i in range(D - 1))
    y = Fraction(x) * Fraction(2) ** (8 * D + 1 - e) + bias
    X = math.floor(y + Fraction(1, 2))
    if y + Fraction(1, 2) == X and X & 1:           # ties to even, of the double 1.5 2^52 + y
        X -= 1
    assert -2 ** 51 <= X < 2 ** 51                   # in the low bits of the FMA's result
    d = [((X >> (8 * i)) & 255) - 128 for i in range(D - 1)] + [X >> (8 * (D - 1))]
    return d[::-1], X - bias


@pytest.mark.parametrize("slices", [4, 5, 6, 8])
@pytest.mark.parametrize("K", [16, 21, 48, 64])
def test_digits(K, slices):
    D = (6 * slices + 7) // 8
    rng = random.Random(100 * K + slices)
    for trial in range(12):
        if trial == 0:      # every digit at its bound
            a = b = [math.nextafter(1.0, 0.0)] * K
        elif trial == 1:
            a, b = [math.nextafter(1.0, 0.0)] * K, [-math.nextafter(1.0, 0.0)] * K
        else:
            a, b = ([rng.gauss(0, 1) * 2.0 ** rng.randrange(-40, 1) for _ in range(K)] for _ in range(2))
        ea, eb = _row_exp(a), _row_exp(b)
        assert all(abs(v) < 2.0 ** (ea - 1) for v in a)
        da, db = [_digits(v, ea, D) for v in a], [_digits(v, eb, D) for v in b]
        for (d, X), v in list(zip(da, a)) + list(zip(db, b)):
            assert sum(t * 256 ** (D - 1 - s) for s, t in enumerate(d)) == X and abs(X) <= 2 ** (8 * D)
            assert abs(d[0]) <= 256 and all(-128 <= t <= 127 for t in d[1:])
        lev = {L: 0 for L in range(D - 4, D + 3)}
        for L in range(2, D + 3):
            terms = [[x[0][s - 1] * y[0][L - s - 1] for s in range(max(1, L - D), min(D, L - 1) + 1)] for x, y in zip(da, db)]
            lev[L] = sum(map(sum, terms))
            assert sum(abs(t) for ts in terms for t in ts) <= 2 ** 23       # every partial sum exact in FP32
            j = L - (D - 4)
            n = 5 if j == 6 else 4 if j == 0 else j + 3                     # units of RP 2^14 in the epilogue
            assert abs(lev[L]) <= n * ((K + 15) // 16 * 16) * 2 ** 14
        w = [lev[L] for L in range(D - 4, D + 3)]
        p1, p2 = w[0] * 256 + w[1], w[2] * 256 + w[3]
        p3 = w[4] * 256 + w[5] + ((w[6] + 128) >> 8)
        assert all(abs(p) < 2 ** 31 for p in (p1, p2, p3))
        acc = (p1 * 65536 + p2) * 65536 + p3
        assert abs(acc) < 2 ** 63
        got = Fraction(acc) * Fraction(2) ** (ea + eb - 8 * (D + 1) - 2)
        want = sum(Fraction(x) * Fraction(y) for x, y in zip(a, b))
        # half a unit of either operand against the other's bound, the dropped levels, the last level's rounding
        bound = K * Fraction(2) ** (ea + eb - 1 - (8 * D + 2)) * (2 + Fraction(1, 64))
        assert abs(got - want) <= bound
