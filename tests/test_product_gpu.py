"""The product on the integer pipes (csrc/soft_mul.cuh) against the FP64 pipe's, bit for bit wherever it
says that it is in its range, and out of range where it has to be."""
import numpy as np
import pytest
import torch

from paper_2510_03932_gb300 import ocp

pytestmark = pytest.mark.gpu


def run(a, b):
    a, b = (np.ascontiguousarray(t, dtype=np.float64) for t in (a, b))
    r, r64, inside = (t.cpu().numpy() for t in ocp.probe_product(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()))
    return r.view(np.int64), r64.view(np.int64), inside == 1.0


def field(v):
    return (v.view(np.int64) >> 52) & 0x7ff


def normal(rng, n, lo, hi, bits=52):
    """Random signs, exponents lo .. hi and significands of `bits` leading bits."""
    frac = rng.integers(0, 1 << bits, n) << (52 - bits)
    return ((rng.integers(lo, hi + 1, n) + 1023) << 52 | frac | rng.integers(0, 2, n) << 63).view(np.float64)


@pytest.mark.parametrize("bits", [52, 26, 27, 3])   # (26, 27: products that end in, or next to, a tie)
@pytest.mark.parametrize("lo,hi", [(-3, 3), (-200, 64), (-500, 500)])
def test_products_of_normal_numbers(bits, lo, hi):
    rng = np.random.default_rng(bits * 1000 + hi)
    a, b = normal(rng, 1 << 20, lo, hi, bits), normal(rng, 1 << 20, lo, hi, bits)
    top = a.view(np.int64) | 0x000fffffffffff00   # significands near two: carries out of the rounding
    for p, q in ((a, b), (top.view(np.float64), b), (top.view(np.float64), (b.view(np.int64) | 0x000ffffffffffff0).view(np.float64))):
        r, r64, inside = run(p, q)
        total = field(p) + field(q) - 2046
        assert np.array_equal(inside, np.abs(total) <= 400)
        assert np.array_equal(r[inside], r64[inside])


def test_special_operands_come_out_of_range():
    rng = np.random.default_rng(5)
    other = np.concatenate([normal(rng, 1 << 16, -600, 600), np.array([0.0, -0.0, 5e-324])])
    for bad in (0.0, -0.0, 5e-324, -1e-310, 2.0 ** -1023):
        for a, b in ((other, np.full_like(other, bad)), (np.full_like(other, bad), other)):
            assert not run(a, b)[2].any()
    other = normal(rng, 1 << 16, -600, 600)   # (the kernels' inputs exclude zeros beside these)
    for bad in (np.inf, -np.inf, np.nan):
        for a, b in ((other, np.full_like(other, bad)), (np.full_like(other, bad), other)):
            assert not run(a, b)[2].any()
