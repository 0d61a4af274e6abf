"""Every shape that ras_setup_shape documents is taken, up to its limit of shared memory and not
beyond, and gives the result of the shape the library picks.

The limit: with the local vectors in shared memory (4 values per point of the box and its ghost
layer), 2048 + 175 x shape[0] x shape[1] x (bytes of a factor value) bytes beside them in 227 KB.
Bars as in the RAS parity tests, between two shapes on the same factors: FP64 max |dz| <= 1e-9
max |z|; FP32 arithmetic 1e-3 in the relative 2-norm.
"""

import dataclasses

import pytest
import torch

from paper_1508_06103_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = {64: (34, 26, 18), 32: (52, 36, 20), 16: (72, 40, 8)}
VALUE = {64: 8, 32: 4, 16: 2}     # bytes of a factor value
VECTOR = {64: 8, 32: 4, 16: 4}    # of a local-vector value
ALL = [(prec, size, held) for prec in SIZES for size in SIZES[prec] for held in (2, 3, 4)]


@pytest.fixture(scope="module")
def api():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1508_06103_gb300 import api as _api
    from paper_1508_06103_gb300 import build

    build.build()
    return _api


def _problem(api, n, levels):
    w = W.random_small(45, cells=(n - 1,) * 3, M=levels - 1, nsens=4, reg="h1l2")
    beta = max(w.h) ** 2
    return api.Problem.from_workload(dataclasses.replace(w, T=(levels - 1) / 16.0, beta1=beta / 100, beta2=beta))


def _close(z, ref, prec):
    if prec == 64:
        return (z - ref).abs().max().item() <= 1e-9 * ref.abs().max().item()
    return torch.linalg.norm(z - ref).item() <= 1e-3 * torch.linalg.norm(ref).item()


def _room(prec, size, held):
    return 227 * 1024 - 2048 - 175 * size * held * VALUE[prec]


@pytest.mark.parametrize("prec, size, held", ALL)
def test_every_size_and_depth_is_taken(api, prec, size, held):
    prob = _problem(api, 6, 7)
    r = torch.from_numpy(W.random_vector(prob.n, 3)).cuda()
    ref = api.RAS(prob, (1, 1, 1, 1), 0, prec).apply(r)
    for place in (0, 2):
        ras = api.RAS(prob, (1, 1, 1, 1), 0, prec, shape=(size, held, 0, place))
        sh = ras.solve_shape()
        assert (sh["chunk_points"], sh["stages"], sh["lanes"]) == (size, held, 4)
        assert _close(ras.apply(r), ref, prec)
        assert ras.status() == 0


@pytest.mark.parametrize("prec, size, held", ALL)
def test_shared_memory_vectors_up_to_the_limit(api, prec, size, held):
    from paper_1508_06103_gb300._lib import KktError

    # the largest box of n x n x n nodes whose vector has room, and one level more, which is refused
    n = 8 if 5 * 1000 * 4 * VECTOR[prec] <= _room(prec, size, held) else 3
    levels = _room(prec, size, held) // ((n + 2) ** 3 * 4 * VECTOR[prec]) - 2
    assert levels >= 2
    prob = _problem(api, n, levels)
    r = torch.from_numpy(W.random_vector(prob.n, 3)).cuda()
    ref = api.RAS(prob, (1, 1, 1, 1), 0, prec).apply(r)
    ras = api.RAS(prob, (1, 1, 1, 1), 0, prec, shape=(size, held, 0, 1))
    sh = ras.solve_shape()
    assert (sh["chunk_points"], sh["stages"], sh["smem_vectors"]) == (size, held, True)
    assert _close(ras.apply(r), ref, prec)
    assert ras.status() == 0
    with pytest.raises(KktError):
        api.RAS(_problem(api, n, levels + 1), (1, 1, 1, 1), 0, prec, shape=(size, held, 0, 1))
