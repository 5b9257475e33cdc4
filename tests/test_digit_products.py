"""The digit arithmetic of the FP64 H*V on the tensor cores (csrc/css_hv_int.cu), restated in Python
integers: seven signed 8-bit digits per entry, products with i + j <= 7, sums exact in FP32."""
from fractions import Fraction

import numpy as np
import pytest

MIN_EXP = 54


def exponents(x):
    """Biased exponents of the entries."""
    return (np.abs(x).view(np.int64) >> 52).astype(int)


def digits(x, shift):
    q = [int(np.rint(v)) for v in np.ldexp(x, shift)]
    out = np.zeros((7, len(q)), dtype=np.int64)
    for k, v in enumerate(q):
        for s in range(6, 0, -1):
            d = (v + 128) % 256 - 128
            out[s, k] = d
            v = (v - d) >> 8
        out[0, k] = v
    return out


def dot(h, v, c=None):
    """Row h of H times column v; c: exponents of the column scales of H (h 2^-c, v 2^c are cut)."""
    c = np.zeros(len(h), int) if c is None else np.maximum(c, -900)
    Eh, Ev = max(exponents(h).max(), MIN_EXP), max((exponents(v) + c).max(), MIN_EXP)
    dh, dv = digits(h, 55 - (Eh - 1022) - c), digits(v, 55 - (Ev - 1022) + c)
    assert np.abs(dh).max() <= 128 and np.abs(dv).max() <= 128
    S = [sum(int(dh[i] @ dv[d - i]) for i in range(7) if 0 <= d - i < 7) for d in range(8)]
    total = sum(s * 256 ** (7 - d) for d, s in enumerate(S))
    return Fraction(total) * Fraction(2) ** int(Eh + Ev - 2 * 1022 - 70)


def exact(h, v):
    return sum(Fraction(float(a)) * Fraction(float(c)) for a, c in zip(h, v))


@pytest.mark.parametrize("K", [8 * 6, 28 * 6, 8 * 23, 28 * 23])
@pytest.mark.parametrize("decades", [0, 12])
def test_error_is_below_the_fp64_sum(K, decades):
    """H v for Gaussian entries, plain or graded (D A D over the decades): summed over 40 rows in units of
    each row's largest term, the digits and the one rounding at the end lose less than an FP64 FMA loop."""
    rng = np.random.default_rng(K)
    d = np.exp2(np.rint(np.linspace(0.0, -decades * np.log2(10.0), K)))
    A = rng.standard_normal((K, K))
    H = A * d[:, None] * d[None, :]
    v = rng.standard_normal(K)
    E = np.maximum(np.array([exponents(r).max() for r in H]), MIN_EXP)
    c = (np.stack([exponents(r) for r in H]) - E[:, None]).max(axis=0)
    err_int = err_fp = Fraction(0)
    for h in H[rng.permutation(K)[:40]]:
        ref = exact(h, v)
        s = Fraction(0)
        for a, x in zip(h, v):  # one rounding of the exact product plus sum
            s = Fraction(float(s + Fraction(float(a)) * Fraction(float(x))))
        unit = Fraction(float(np.abs(h * v).max()))
        err_int += abs(Fraction(float(dot(h, v, c))) - ref) / unit
        err_fp += abs(s - ref) / unit
    assert err_int < err_fp


@pytest.mark.parametrize("scale_h,scale_v", [(0, 0), (-300, 200), (900, -900), (-1000, 0), (-1070, 1000), (960, 0)])
def test_exponent_range(scale_h, scale_v):
    """Powers of two up to the ends of the FP64 range: entries keep 2^-56 of their vector's largest, or
    2^-1023 where that is below the smallest digit."""
    rng = np.random.default_rng(1)
    h, v = np.ldexp(rng.standard_normal(30), scale_h), np.ldexp(rng.standard_normal(30), scale_v)
    hm, vm = Fraction(float(np.abs(h).max())), Fraction(float(np.abs(v).max()))
    eh = max(2 * hm / Fraction(2) ** 56, Fraction(1, 2 ** 1023))
    ev = max(2 * vm / Fraction(2) ** 56, Fraction(1, 2 ** 1023))
    bound = 30 * (eh * vm + ev * hm + eh * ev + 4 * hm * vm / Fraction(2) ** 61)
    assert abs(dot(h, v) - exact(h, v)) <= bound


@pytest.mark.parametrize("b", range(1, 25))
def test_sums_stay_exact_in_fp32(b):
    """At most seven products of 146 // b blocks of b digits of magnitude 128 are summed."""
    assert 7 * (146 // b) * b * 128 * 128 < 2 ** 24
