"""One-level RAS applies (ILU(0)) on boxes at the edges of the solve's and the factorisation's
shapes, against the oracle's ILU(0) RAS: wavefronts with no point and with one, ragged groups of
8 points, more and fewer groups than warps, boxes of one node, single points beside long axes,
more wavefronts than the solve keeps pointers of in shared memory.

Bars as in the other RAS parity tests: FP64 max |dz| <= 1e-9 max |z| (same pattern and IKJ order,
rounding order only), FP32 factors 1e-3 and BF16-stored factors 8 * 2^-8 in the relative 2-norm.
"""

import dataclasses

import numpy as np
import pytest
import torch

from oracle import kkt as okkt
from oracle import schwarz as osch
from paper_1508_06103_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# cells, M, nsub, overlap
CASES = {
    "one-node-boxes": ((2, 1, 1), 2, (3, 2, 2, 3), 0),
    "x-line": ((17, 1, 1), 2, (2, 1, 1, 1), 1),
    "t-line": ((1, 1, 1), 21, (1, 1, 1, 2), 1),
    "flat-x": ((1, 6, 5), 6, (2, 1, 1, 1), 0),
    "cube-ov2": ((6, 5, 6), 7, (2, 1, 2, 2), 2),
    "wide-wavefronts": ((10, 9, 9), 8, (1, 1, 1, 1), 0),
    "many-wavefronts": ((1, 1, 1), 1030, (1, 1, 1, 1), 0),
}


@pytest.fixture(scope="module")
def api():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1508_06103_gb300 import api as _api
    from paper_1508_06103_gb300 import build

    build.build()
    return _api


@pytest.fixture(scope="module")
def oracle():
    done = {}

    def get(name):
        if name not in done:
            cells, M, nsub, ov = CASES[name]
            # H1-L2 where the box is (nearly) the whole grid in space: the H1-H1 regulariser has the
            # constant source in its null space, its last pivot is rounding, and z is 1e15
            reg = "h1l2" if name in ("flat-x", "many-wavefronts") else "h1h1"
            w = W.random_small(41, cells=cells, M=M, nsens=4, reg=reg)
            # beta as in the 32^3 x 64 family, beta2 ~ h^2: ILU(0) grows without bound at smaller ratios
            beta = max(w.h) ** 2
            w = dataclasses.replace(w, T=M / 16.0, beta1=beta / 100, beta2=beta)
            p = okkt.Problem.from_workload(w)
            r = W.random_vector(p.N * p.L * 3, 5)
            done[name] = w, r, osch.RAS(p, okkt.assemble(p), nsub, ov, "ilu0").apply(r)
        return done[name]

    return get


@pytest.mark.parametrize("prec", [64, 32, 16])
@pytest.mark.parametrize("name", CASES)
def test_ras_apply_on_edge_shapes_matches_oracle(api, oracle, name, prec):
    _, _, nsub, ov = CASES[name]
    w, r, zr = oracle(name)
    prob = api.Problem.from_workload(w)
    ras = api.RAS(prob, nsub, ov, prec)
    for _ in range(2):   # the second pass after a refactorisation in place
        z = ras.apply(torch.from_numpy(r).cuda()).cpu().numpy()
        if prec == 64:
            assert np.abs(z - zr).max() <= 1e-9 * np.abs(zr).max()
        else:
            assert np.linalg.norm(z - zr) <= (1e-3 if prec == 32 else 8 * 2.0**-8) * np.linalg.norm(zr)
        ras.refactor()


# exact local LU: bands within one CTA's threads and beyond, fewer unknowns than threads
LU_CASES = {
    "few-unknowns": ((1, 1, 1), 3, (1, 1, 1, 1), 0),
    "band-in-one-pass": ((5, 5, 6), 3, (1, 1, 1, 1), 0),
    "band-over-one-pass": ((6, 6, 7), 3, (1, 1, 1, 1), 0),
}


@pytest.mark.parametrize("name", LU_CASES)
def test_exact_lu_on_edge_shapes_matches_oracle(api, name):
    # bar: 100 cond_1 u max|z|, as in test_gpu_solve.py (both sides backward stable)
    cells, M, nsub, ov = LU_CASES[name]
    w = W.random_small(43, cells=cells, M=M, nsens=4, reg="h1l2")
    beta = max(w.h) ** 2
    w = dataclasses.replace(w, T=M / 16.0, beta1=beta / 100, beta2=beta)
    p = okkt.Problem.from_workload(w)
    F = okkt.assemble(p)
    ref = osch.RAS(p, F, nsub, ov, "lu")
    kappa = max(np.linalg.cond(F[idx][:, idx].toarray(), 1) for idx in ref.idx)
    prob = api.Problem.from_workload(w)
    ras = api.RAS(prob, nsub, ov, 64, local="lu")
    for seed in (1, 2):
        r = W.random_vector(prob.n, seed)
        z, zr = ras.apply(torch.from_numpy(r).cuda()).cpu().numpy(), ref.apply(r)
        assert np.abs(z - zr).max() <= 100 * kappa * 2.0**-53 * np.abs(zr).max()


# boxes solved by one CTA, by a cluster of 2, 4 and 8 CTAs (FP64; FP32 and BF16: 1, 1, 4, 8)
CLUSTER_CELLS = {"2": (10, 9, 9, 8), "4": (20, 11, 8, 6), "8": (27, 15, 9, 6)}


@pytest.mark.parametrize("prec", [64, 32, 16])
@pytest.mark.parametrize("name", CLUSTER_CELLS)
def test_box_shared_by_ctas_has_the_bits_of_one_cta(api, name, prec):
    # the same groups with the same operations in the same order: no tolerance.  Enough copies of
    # the problem in one batch leave every box to a CTA of its own.
    *cells, M = CLUSTER_CELLS[name]
    w = W.random_small(44, cells=tuple(cells), M=M, nsens=4, reg="h1l2")
    beta = max(w.h) ** 2
    w = dataclasses.replace(w, T=M / 16.0, beta1=beta / 100, beta2=beta)
    probs = [api.Problem.from_workload(w) for _ in range(80)]
    many = api.BatchRAS(probs, (1, 1, 1, 1), 0, prec)
    one = api.RAS(probs[0], (1, 1, 1, 1), 0, prec)
    r = torch.from_numpy(W.random_vector(probs[0].n, 6)).cuda()
    z = one.apply(r)
    assert torch.isfinite(z).all() and z.abs().max() > 0
    assert torch.equal(many.apply(r.repeat(80))[-probs[0].n:], z)
    assert one.status() == 0


# the forms the chooser takes: clusters for the few boxes above, one CTA a box for many of them
@pytest.mark.parametrize("prec", [64, 32, 16])
@pytest.mark.parametrize("name", CLUSTER_CELLS)
def test_few_boxes_take_a_cluster_and_many_do_not(api, name, prec):
    *cells, M = CLUSTER_CELLS[name]
    w = W.random_small(44, cells=tuple(cells), M=M, nsens=4, reg="h1l2")
    beta = max(w.h) ** 2
    w = dataclasses.replace(w, T=M / 16.0, beta1=beta / 100, beta2=beta)
    probs = [api.Problem.from_workload(w) for _ in range(80)]
    form = api.RAS(probs[0], (1, 1, 1, 1), 0, prec).solve_form()
    assert form["cluster"] == (1 if prec != 64 and name == "2" else int(name)) and not form["ring"]
    form = api.BatchRAS(probs, (1, 1, 1, 1), 0, prec).solve_form()
    # the ring of "8" (508 points in a wavefront) beside 16 FP32 buffers would take 233,104 of 232,448 bytes
    assert form["cluster"] == 1 and form["ring"] == (prec == 16 or (prec == 32 and name != "8"))


# the ring of wavefronts in shared memory is taken from a quarter as many boxes as SMs: enough
# copies of the problem in one batch
@pytest.mark.parametrize("prec", [32, 16])
@pytest.mark.parametrize("name", CASES)
def test_ring_of_wavefronts_on_edge_shapes_matches_oracle(api, oracle, name, prec):
    _, _, nsub, ov = CASES[name]
    w, r, zr = oracle(name)
    copies = -(-40 // int(np.prod(nsub)))
    probs = [api.Problem.from_workload(w) for _ in range(copies)]
    ras = api.BatchRAS(probs, nsub, ov, prec)
    form = ras.solve_form()
    assert form["ring"] and form["cluster"] == 1 and form["buffers"] >= 1
    z = ras.apply(torch.from_numpy(r).cuda().repeat(copies)).view(copies, -1)
    assert torch.equal(z, z[:1].expand_as(z))
    z0 = z[0].cpu().numpy()
    assert np.linalg.norm(z0 - zr) <= (1e-3 if prec == 32 else 8 * 2.0**-8) * np.linalg.norm(zr)
    assert ras.status() == 0
