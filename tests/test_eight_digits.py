"""The eight-digit arithmetic of the FP64 H*V on the tensor cores (csrc/css_hv_int.cu), restated in Python
integers: eight signed 8-bit digits per entry, products with i + j <= 8, sums exact in FP32 and 64 bits."""
from fractions import Fraction

import numpy as np
import pytest

MIN_EXP, DIGITS, BITS = 61, 8, 62


def exponents(x):
    """Biased exponents of the entries."""
    return (np.abs(x).view(np.int64) >> 52).astype(int)


def digits(x, shift):
    out = np.zeros((DIGITS, len(x)), dtype=np.int64)
    for k, v in enumerate(int(np.rint(v)) for v in np.ldexp(x, shift)):
        assert abs(v) <= 2 ** BITS
        for s in range(DIGITS - 1, 0, -1):
            d = (v + 128) % 256 - 128
            out[s, k] = d
            v = (v - d) >> 8
        out[0, k] = v
    assert np.abs(out[0]).max() <= 65 and np.abs(out).max() <= 128
    return out


def dot(h, v):
    """Row h of H times column v, both scaled by their largest entries."""
    Eh, Ev = max(exponents(h).max(), MIN_EXP), max(exponents(v).max(), MIN_EXP)
    dh, dv = digits(h, BITS - (Eh - 1022)), digits(v, BITS - (Ev - 1022))
    S = [sum(int(dh[i] @ dv[d - i]) for i in range(DIGITS) if 0 <= d - i < DIGITS) for d in range(DIGITS + 1)]
    hi = sum(S[d] * 256 ** (4 - d) for d in range(5))
    lo = sum(S[d] * 256 ** (8 - d) for d in range(5, 9))
    assert max(abs(hi), abs(lo)) < 2 ** 63
    return Fraction(hi * 2 ** 32 + lo) * Fraction(2) ** int(Eh + Ev - 2 * 1022 - 76)


def exact(h, v):
    return sum(Fraction(float(a)) * Fraction(float(c)) for a, c in zip(h, v))


def bound(h, v):
    """Rounding of the entries to 2^-63 of the power of two above the largest (2^-1024 when that is below the
    smallest digit) and the 21 products that are left out, below 2^-69 of it each."""
    n, hm, vm = len(h), Fraction(float(np.abs(h).max())), Fraction(float(np.abs(v).max()))
    eh = max(2 * hm / Fraction(2) ** 63, Fraction(1, 2 ** 1024))
    ev = max(2 * vm / Fraction(2) ** 63, Fraction(1, 2 ** 1024))
    sh, sv = eh * 2 ** 63, ev * 2 ** 63
    return n * (eh * vm + ev * hm + eh * ev + 21 * sh * sv / Fraction(2) ** 69)


@pytest.mark.parametrize("K", [1, 6, 28 * 6, 28 * 23])
@pytest.mark.parametrize("scale_h,scale_v", [(0, 0), (-300, 200), (900, -900), (-1000, 0), (-1070, 1000), (960, 0)])
def test_error_bound_over_the_exponent_range(K, scale_h, scale_v):
    rng = np.random.default_rng(K)
    h, v = np.ldexp(rng.standard_normal(K), scale_h), np.ldexp(rng.standard_normal(K), scale_v)
    assert abs(dot(h, v) - exact(h, v)) <= bound(h, v)


@pytest.mark.parametrize("K", [6, 28 * 23])
def test_digits_at_their_limits(K):
    """Entries next to powers of two, whose digits round up into the next one, and constant ones, whose sums grow."""
    for x in (np.nextafter(1.0, 0.0), -np.nextafter(1.0, 0.0), 0.5 - 2.0 ** -54, 0.501953125 - 2.0 ** -10):
        h, v = np.full(K, x), np.full(K, -x)
        assert abs(dot(h, v) - exact(h, v)) <= bound(h, v)


@pytest.mark.parametrize("b", range(1, 25))
def test_sums_stay_exact_in_fp32(b):
    """145 // b blocks of b terms: the sum d = 7 takes six products of two digits up to 128 and two with the
    leading digit, up to 65; d = 8 seven without it."""
    K = 145 // b * b
    assert K * (6 * 128 * 128 + 2 * 65 * 128) < 2 ** 24 and K * 7 * 128 * 128 < 2 ** 24
