"""The fixed-point slicing of a float pair (tc_gemm.cuh, slice_fields and
slice_pack) restated in numpy: digits within [-64, 64], and the rest after four
slices within 1.01 2^-29 of the value."""
from fractions import Fraction

import numpy as np
import pytest

F, U = np.float32, np.uint32


def slices(hi, lo):
    a = hi + F(768)
    rest = hi - (a - F(768))
    b = (rest + lo) + F(0.046875)
    bias = 64 * (1 + (1 << 7) + (1 << 14) + (1 << 21))
    with np.errstate(over="ignore"):
        u = (a.view(U) << U(14)) + b.view(U) + U((bias - (0x44400000 << 14) - 0x3D400000) % (1 << 32))
    out = []
    for p in range(4):
        f = (u >> U(7 * (3 - p))) & U(0xFF if p == 0 else 0x7F)
        v = ((f | U(0x4300)) << U(16)).view(F)               # the BF16 of these bits
        out.append((v - F(192)).astype(np.int64))
    return out


@pytest.mark.parametrize("scale", [0.49999997, 0.25, 2.0 ** -7, 2.0 ** -14, 2.0 ** -20, 2.0 ** -28, 2.0 ** -60, 0.0])
def test_slices(scale):
    rng = np.random.default_rng(3)
    hi = (rng.uniform(-1, 1, 4000) * scale).astype(F)
    hi[:6] = F(scale) * np.array([1, -1, 0.5, -0.5, 0, 1 / 128], F)
    lo = (rng.uniform(-0.5, 0.5, 4000) * np.spacing(np.abs(hi))).astype(F)
    lo[0] = lo[1] = 0
    d = slices(hi, lo)
    for q in d:
        assert np.abs(q).max() <= 64
    for k in range(4000):
        got = sum(Fraction(int(d[p][k]), 128 ** (p + 1)) for p in range(4))
        assert abs(Fraction(float(hi[k])) + Fraction(float(lo[k])) - got) <= Fraction(101, 100) / 2 ** 29


def test_every_half_integer_edge():
    """Values at and beside the digits' rounding edges."""
    k = np.arange(-128, 129)
    for step in (2.0 ** -8, 2.0 ** -15, 2.0 ** -22, 2.0 ** -29):
        hi = (k * step).astype(F)
        hi = hi[np.abs(hi) <= 0.5]
        for lo in (np.zeros_like(hi), np.spacing(hi) / F(2), -np.spacing(hi) / F(4)):
            d = slices(hi, lo)
            assert max(np.abs(q).max() for q in d) <= 64
            got = sum(q.astype(np.float64) / 128.0 ** (p + 1) for p, q in enumerate(d))
            assert np.abs(hi.astype(np.float64) + lo - got).max() <= 1.01 * 2.0 ** -29
