"""The division of the exact local LU's backward sweep against CUDA's division.

Bars: the same bits where values and quotients are normal numbers (the corrected quotient is
rounded correctly); one unit in the last place where one of them is subnormal; infinities, zeros
and NaN as the division gives them.
"""

import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def quotient():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1508_06103_gb300 import _lib, build

    build.build()

    def run(v, d):
        q = torch.empty_like(v)
        assert _lib.load().lu_selftest_quotient(ctypes.c_void_p(v.data_ptr()), ctypes.c_void_p(d.data_ptr()),
                                                ctypes.c_void_p(q.data_ptr()), v.numel(), None) == 0
        torch.cuda.synchronize()
        return q

    return run


def _values(n, seed, lo, hi):
    g = torch.Generator("cuda").manual_seed(seed)
    m = 1 + torch.rand(n, dtype=torch.float64, device="cuda", generator=g)
    e = torch.randint(lo, hi + 1, (n,), device="cuda", generator=g).double()
    s = 1 - 2 * torch.randint(0, 2, (n,), device="cuda", generator=g).double()
    half = torch.floor(e / 2)
    return s * m * torch.exp2(half) * torch.exp2(e - half)


@pytest.mark.parametrize("lo, hi, ulps", [(-3, 3, 0), (-500, 500, 0), (-1060, 1022, 1)])
def test_quotient_has_the_bits_of_the_division(quotient, lo, hi, ulps):
    n = 1 << 22
    v, d = _values(n, 1, lo, hi), _values(n, 2, lo, hi)
    q, ref = quotient(v, d), v / d
    same = (q == ref) | (q.isnan() & ref.isnan())
    if ulps:
        same |= q.isfinite() & ref.isfinite() & ((q.view(torch.int64) - ref.view(torch.int64)).abs() <= ulps)
    assert same.all()


def test_quotient_of_zeros_infinities_and_nan(quotient):
    s = torch.tensor([0.0, -0.0, 1.0, -2.0, 5e-324, 1.7e308, float("inf"), float("-inf"), float("nan")],
                     dtype=torch.float64, device="cuda")
    v, d = (t.reshape(-1).contiguous() for t in torch.meshgrid(s, s, indexing="ij"))
    q, ref = quotient(v, d), v / d
    assert ((q == ref) | (q.isnan() & ref.isnan())).all()
