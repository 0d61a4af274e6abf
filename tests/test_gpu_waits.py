"""The subdomain solve's bounded waits when they run out: one verdict per warp.

Every wait ends (limits of milliseconds), every kernel returns, and after ras_refactor the handle
gives the bits it gave before.
"""

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
