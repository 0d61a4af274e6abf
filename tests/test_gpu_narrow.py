"""ILU(0) subdomains of a few points a wavefront (lines, thin plates, a few nodes a side): their
factors are stored in narrow groups, against the oracle's ILU(0) RAS and a bound on their size.

Bars as in the other RAS parity tests: FP64 max |dz| <= 1e-9 max |z|, FP32 factors 1e-3 and
BF16-stored factors 8 * 2^-8 in the relative 2-norm.
"""

import dataclasses

import numpy as np
import pytest
import torch

from oracle import kkt as okkt
from oracle import schwarz as osch
from paper_1508_06103_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# nodes and levels, split, overlap
CASES = {
    "x-lines": ((17, 2, 3, 4), (1, 2, 3, 4), 0),
    "t-lines": ((3, 3, 2, 40), (3, 3, 2, 1), 0),
    "cubes-2": ((4, 4, 4, 4), (2, 2, 2, 2), 0),
    "cubes-3": ((9, 9, 9, 9), (3, 3, 3, 3), 0),
    "cubes-3-and-4": ((8, 8, 8, 9), (4, 4, 4, 4), 1),
    "xt-plates": ((17, 2, 2, 25), (1, 2, 2, 1), 0),
    "xy-plates": ((8, 8, 2, 2), (1, 1, 2, 2), 0),
}


@pytest.fixture(scope="module")
def api():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1508_06103_gb300 import api as _api
    from paper_1508_06103_gb300 import build

    build.build()
    return _api


def _problem(dims):
    w = W.random_small(46, cells=tuple(n - 1 for n in dims[:3]), M=dims[3] - 1, nsens=4)
    beta = max(w.h) ** 2
    return dataclasses.replace(w, T=(dims[3] - 1) / 16.0, beta1=beta / 100, beta2=beta)


def _wavefronts(dims, nsub, overlap):
    """Points of every wavefront of every box."""
    axes = []
    for n, p in zip(dims, nsub):
        cut = np.cumsum([0] + [n // p + (k < n % p) for k in range(p)])
        axes.append([min(n, cut[k + 1] + overlap) - max(0, cut[k] - overlap) for k in range(p)])
    for lx in axes[0]:
        for ly in axes[1]:
            for lz in axes[2]:
                for lt in axes[3]:
                    t, z, y, x = np.meshgrid(*(range(v) for v in (lt, lz, ly, lx)), indexing="ij")
                    yield np.bincount((x + 2 * y + 4 * z + 8 * t).ravel())


@pytest.mark.parametrize("prec", [64, 32, 16])
@pytest.mark.parametrize("name", CASES)
def test_narrow_boxes_match_oracle(api, name, prec):
    dims, nsub, ov = CASES[name]
    w = _problem(dims)
    p = okkt.Problem.from_workload(w)
    prob = api.Problem.from_workload(w)
    r = W.random_vector(prob.n, 5)
    zr = osch.RAS(p, okkt.assemble(p), nsub, ov, "ilu0").apply(r)
    for place in (0, 1, 2):   # as chosen, local vectors in shared and in global memory
        ras = api.RAS(prob, nsub, ov, prec, shape=(0, 0, 0, place))
        for _ in range(2):   # the second pass after a refactorisation in place
            z = ras.apply(torch.from_numpy(r).cuda()).cpu().numpy()
            if prec == 64:
                assert np.abs(z - zr).max() <= 1e-9 * np.abs(zr).max()
            else:
                assert np.linalg.norm(z - zr) <= (1e-3 if prec == 32 else 8 * 2.0**-8) * np.linalg.norm(zr)
            ras.refactor()
        assert ras.status() == 0


@pytest.mark.parametrize("prec", [64, 32, 16])
@pytest.mark.parametrize("name", CASES)
def test_narrow_boxes_take_no_more_than_a_third_beyond_short_rows(api, name, prec):
    # the yardstick: a wavefront's rows padded to 2 points in FP64 (4 in FP32, 8 in BF16) when it has no
    # more, to the next 8 k + 2 (16 k + 4, 32 k + 8) when it has
    dims, nsub, ov = CASES[name]
    first, step = {64: (2, 8), 32: (4, 16), 16: (8, 32)}[prec]
    places = boxes = 0
    for h in _wavefronts(dims, nsub, ov):
        boxes += 1
        places += sum(first + max(0, -(-(int(n) - first) // step)) * step for n in h if n)
    values = api.RAS(api.Problem.from_workload(_problem(dims)), nsub, ov, prec).info()["factor_values"]
    # 328 values a point in FP32 and BF16 (2 places unused), a unit row a box in FP64
    assert values <= 4 / 3 * places * (326 if prec == 64 else 328) + (boxes * 326 * 2 if prec == 64 else 0)


# many boxes of one group a wavefront: CTAs of fewer warps than the smallest size class has
@pytest.mark.parametrize("prec", [64, 32, 16])
@pytest.mark.parametrize("dims, nsub", [((17, 17, 17, 9), (1, 17, 17, 9)), ((18, 18, 18, 18), (6, 6, 6, 6))],
                         ids=["lines", "cubes"])
def test_many_narrow_boxes_take_fewer_warps(api, dims, nsub, prec):
    w = _problem(dims)
    prob = api.Problem.from_workload(w)
    ras = api.RAS(prob, nsub, 0, prec)
    assert ras.solve_form()["warps"] in (1, 2, 3)
    # the same groups in the same order on 16 warps: the same bits (16 warps are held to the oracle elsewhere)
    few = api.RAS(prob, nsub, 0, prec, shape=({64: 34, 32: 52, 16: 72}[prec], 0, 0, 2))
    assert few.solve_form()["warps"] == 16
    r = torch.from_numpy(W.random_vector(prob.n, 5)).cuda()
    z = ras.apply(r)
    assert torch.isfinite(z).all() and z.abs().max() > 0 and torch.equal(z, few.apply(r))
    assert ras.status() == 0
