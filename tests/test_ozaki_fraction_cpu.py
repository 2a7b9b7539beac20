"""The reconstruction of the modular Ozaki GEMM (csrc/gemm_oz.cu, oz_crt_rows) emulated with Python integers, no
device needed: F = sum_g w_g round(2^88 / p_t) modulo 2^88 over the (modulus, chunk) groups is x / P in units of 2^-88
up to sum |w| / 2 units, for every |x| <= P / 4 and residues as the GEMM leaves them (|w| <= 65 a chunk, not reduced into
the balanced range); an exact zero comes back within the snapping threshold; the byte sums and their pairs stay
inside the integer ranges the kernel uses."""
import random

import pytest

from tests.test_ozaki_scheme_cpu import MODULI

FL = 11


def _value(x, T, nch, rng):
    """(F, sum |w|, byte sums) for the integer x."""
    P = 1
    for p in MODULI[:T]:
        P *= p
    F, ws, sums = 0, 0, [0] * FL
    for p in MODULI[:T]:
        w = x * pow(P // p, -1, p) % p
        parts = [rng.randrange(-60, 61) for _ in range(nch - 1)]
        last = (w - sum(parts)) % p
        last -= p if last > p // 2 else 0
        if rng.random() < 0.2 and abs(last - p) <= 65:      # a residue past the balanced range
            last -= p
        parts.append(last)
        assert all(abs(v) <= 65 for v in parts)
        C = (2 ** 88 + p // 2) // p
        for v in parts:
            ws += abs(v)
            F += v * C
            for l in range(FL):
                sums[l] += v * ((C >> (8 * l)) & 255)
    assert sum(s << (8 * l) for l, s in enumerate(sums)) == F
    return F, ws, sums, P


@pytest.mark.parametrize("nch", [1, 2])
@pytest.mark.parametrize("T", [9, 13, 16, 17, 19])
def test_fraction_is_x_over_P(T, nch):
    rng = random.Random(100 * T + nch)
    P = _value(0, T, nch, rng)[3]
    for k in range(200):
        x = [0, 1, -1, P // 4, -(P // 4)][k] if k < 5 else rng.randrange(-(P // 4), P // 4 + 1) >> rng.randrange(0, 90)
        F, ws, sums, _ = _value(x, T, nch, rng)
        f = F % 2 ** 88
        f -= 2 ** 88 if f >= 2 ** 87 else 0                  # signed
        err = abs(f * P - x * 2 ** 88)                       # in units of P 2^-88 / P
        assert err <= (ws * P) // 2 + P
        assert ws <= 19 * nch * 65
        if x == 0:
            assert abs(f) * 256 < 2 ** 19                    # snapped to zero (the kernel works on 2^8 F)
        for l in range(FL):
            assert abs(sums[l]) < 2 ** 21                    # pairs a + 256 b within 32 bits
