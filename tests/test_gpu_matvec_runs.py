"""FP64 KKT matvec and residual where tiles and level runs end, against the oracle's assembled F_h.

Grids of one cell, of exactly one tile and of one node more, ragged tiles, one step, runs of one
level (few tiles) and of several with a ragged last one (many tiles), both regularisers, both time
schemes.  Bar: |y - y_ref| <= 1e-12 (|F||x|)_i per output, as in test_gpu_kkt.py (each side's
rounding is below 330 u (|F||x|)_i).
"""

import numpy as np
import pytest
import torch

from oracle import kkt as okkt
from paper_1508_06103_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# cells, M
CASES = [((1, 1, 1), 1), ((2, 1, 1), 2), ((10, 10, 2), 3), ((11, 11, 3), 1), ((7, 7, 3), 5), ((22, 21, 10), 25),
         ((1, 1, 1), 300)]


@pytest.fixture(scope="module")
def api():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1508_06103_gb300 import api as _api
    from paper_1508_06103_gb300 import build

    build.build()
    return _api


@pytest.mark.parametrize("reg,theta", [("h1h1", 0.5), ("h1l2", 1.0)])
@pytest.mark.parametrize("cells,M", CASES, ids=[f"{'x'.join(map(str, c))}x{m}" for c, m in CASES])
def test_fp64_matvec_and_residual_match_oracle(api, cells, M, reg, theta):
    w = W.random_small(51, cells=cells, M=M, theta=theta, reg=reg, nsens=5,
                       dirichlet_faces=W.FACE_X0 if max(cells) > 1 else W.FACE_Z1)
    p = okkt.Problem.from_workload(w)
    F = okkt.assemble(p)
    prob = api.Problem.from_workload(w)
    x, b = W.random_vector(prob.n, 3), W.random_vector(prob.n, 4)
    bound = 1e-12 * (abs(F) @ np.abs(x)) + 1e-300
    xd, bd = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    y = prob.apply(xd).cpu().numpy()
    assert np.all(np.abs(y - F @ x) <= bound)
    r = prob.residual(bd, xd).cpu().numpy()
    assert np.all(np.abs(r - (b - F @ x)) <= bound + 1e-15 * np.abs(b))


def test_enqueueing_does_not_grow_with_the_levels(api):
    # a call is one launch (some 8 us of host time); looking at every run length of 9000 levels took 110 us
    import time

    prob = api.Problem.from_workload(W.random_small(52, cells=(2, 2, 2), M=9000, nsens=2))
    x = torch.from_numpy(W.random_vector(prob.n, 3)).cuda()
    y = torch.empty_like(x)
    times = []
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(20):
            prob.apply(x, out=y)
        times.append((time.perf_counter() - t) / 20)
    torch.cuda.synchronize()
    assert min(times) < 50e-6
