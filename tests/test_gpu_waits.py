"""The subdomain solve's bounded waits when they run out: one verdict per warp, and every copy into
shared memory waited for before a CTA leaves, and none of a box's CTAs writes z.

Every wait ends (limits of milliseconds), every kernel returns, and after ras_refactor the handle
gives the bits it gave before.
"""

import dataclasses
import time

import numpy as np
import pytest
import torch

from paper_1508_06103_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1508_06103_gb300 import api as _api
    from paper_1508_06103_gb300 import build

    build.build()
    return _api


@pytest.mark.parametrize("kind", [0, 1], ids=["mbarrier", "counter"])
def test_lanes_of_a_warp_get_one_verdict(api, kind):
    from paper_1508_06103_gb300._lib import KktError

    w = W.random_small(41, cells=(5, 4, 3), M=5, nsens=4)
    prob = api.Problem.from_workload(w)
    ras = api.RAS(prob, (2, 2, 1, 2), 1, 32)
    r = torch.from_numpy(W.random_vector(prob.n, 3)).cuda()
    z0 = ras.apply(r).clone()
    assert ras.selftest_lanes(kind) == [0] * 32   # the shorter limit of half of the lanes ends it for all
    with pytest.raises(KktError) as e:
        ras.status()
    assert e.value.status == -3
    ras.refactor()
    assert ras.status() == 0 and torch.equal(ras.apply(r), z0)


def _groups(dims, nsub, overlap):
    """Groups of 8 points of every box of the split (boxes of uneven parts, overlap trimmed)."""
    axes = []
    for n, p in zip(dims, nsub):
        cut = np.cumsum([0] + [n // p + (k < n % p) for k in range(p)])
        axes.append([min(n, cut[k + 1] + overlap) - max(0, cut[k] - overlap) for k in range(p)])
    for lx in axes[0]:
        for ly in axes[1]:
            for lz in axes[2]:
                for lt in axes[3]:
                    t, z, y, x = np.meshgrid(*(range(v) for v in (lt, lz, ly, lx)), indexing="ij")
                    yield sum(-(-int(c) // 8) for c in np.bincount((x + 2 * y + 4 * z + 8 * t).ravel()))


@pytest.mark.parametrize("dims, nsub, place", [((6, 5, 4, 6), (2, 2, 1, 2), 1), ((6, 5, 4, 6), (2, 2, 1, 2), 2),
                                               ((12, 10, 8, 16), (3, 2, 2, 4), 2)],
                         ids=["vectors-in-smem", "plain", "ring"])
@pytest.mark.parametrize("stages", [2, 3, 4])
def test_a_solve_that_gives_up_waits_for_its_copies(api, stages, dims, nsub, place):
    # every warp gives up at its first group: that one's copy has landed, the next `buffers` groups'
    # are in flight
    from paper_1508_06103_gb300._lib import KktError

    w = W.random_small(41, cells=tuple(n - 1 for n in dims[:3]), M=dims[3] - 1, nsens=4)
    prob = api.Problem.from_workload(w)
    ras = api.RAS(prob, nsub, 1, 32, shape=(20, stages, 0, place))
    form = ras.solve_form()
    assert form["cluster"] == 1 and form["ring"] == (nsub[0] == 3) and form["buffers"] == stages - 1
    r = torch.from_numpy(W.random_vector(prob.n, 3)).cuda()
    z0 = ras.apply(r).clone()
    z = torch.full_like(r, 7.0)
    expect = 0
    for ng in _groups(dims, nsub, 1):
        expect += sum(range(form["warps"] + 1, min(2 * ng, (form["buffers"] + 1) * form["warps"]) + 1))
    assert ras.selftest_solve(r, z, 5.0) == expect > 0
    assert (z == 7.0).all()
    with pytest.raises(KktError) as e:
        ras.status()
    assert e.value.status == -3
    ras.refactor()
    assert ras.status() == 0 and torch.equal(ras.apply(r), z0)


@pytest.mark.parametrize("cta", [0, 1, 3])
@pytest.mark.parametrize("hold", [1, 2], ids=["counter", "copies"])
def test_one_cta_that_gives_up_ends_its_whole_cluster(api, hold, cta):
    # the other CTAs keep the 2 s limit, so a return within a second means that they were told
    from paper_1508_06103_gb300._lib import KktError

    w = W.random_small(44, cells=(20, 11, 8), M=6, nsens=4, reg="h1l2")
    beta = max(w.h) ** 2
    w = dataclasses.replace(w, T=6 / 16.0, beta1=beta / 100, beta2=beta)
    prob = api.Problem.from_workload(w)
    ras = api.RAS(prob, (1, 1, 1, 1), 0, 32)
    assert ras.solve_form()["cluster"] == 4
    r = torch.from_numpy(W.random_vector(prob.n, 3)).cuda()
    z0 = ras.apply(r).clone()
    z = torch.full_like(r, 7.0)
    torch.cuda.synchronize()
    t = time.perf_counter()
    ras.selftest_solve(r, z, 5.0, hold=hold, cta=cta)
    assert time.perf_counter() - t < 1.0
    assert (z == 7.0).all()
    with pytest.raises(KktError) as e:
        ras.status()
    assert e.value.status == -3
    ras.refactor()
    assert ras.status() == 0 and torch.equal(ras.apply(r), z0)
