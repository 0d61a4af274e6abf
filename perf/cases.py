"""The work that users of this package have it do, as cases to be timed and compared.

A case goes through the Python binding (`paper_1508_06103_gb300.api`): the KKT matvec, one-level
RAS applies with every local solver and precision, refactorisation with a two-level apply, and
whole solves (one problem, and several together).  Meshes, splits, overlaps and solver settings
are those of the package's workloads, tests and benchmark, or lie between them.

`exact` forms the same operators in 64 bits with plain torch: the finite elements by quadrature,
F_h row by row, incomplete factorisations by wavefronts over the points of all boxes at once.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1508_06103_gb300 import api

LENGTHS = (1.0, 1.0, 1.0)
FACES = 1                    # Dirichlet on x = 0, the benchmark's
DIRICHLET_ALL = 63           # the smallest workload's
MID = dict(cx=32, cy=32, cz=32, M=64)          # the benchmark's mesh
MID_SPLIT = dict(px=4, py=4, pz=4, pt=4, overlap=2)
VALUE_BYTES = {64: 8, 32: 4, 16: 2}
ITERATIONS = 20              # outer iterations of a two-level solve to 1e-8, about


def _apply(name, cells, M, prec, elem="q1", reg="h1h1", theta=0.5, faces=FACES):
    return dict(name=name, kind="apply", cx=cells[0], cy=cells[1], cz=cells[2], M=M, prec=prec, elem=elem, reg=reg,
                theta=theta, faces=faces)


def _ras(name, kind, cells, M, split, overlap, prec, local="ilu0", theta=0.5, faces=FACES, elem="q1", reg="h1h1"):
    return dict(name=name, kind=kind, cx=cells[0], cy=cells[1], cz=cells[2], M=M, px=split[0], py=split[1],
                pz=split[2], pt=split[3], overlap=overlap, prec=prec, local=local, theta=theta, faces=faces, elem=elem,
                reg=reg)


def _batch(name, first, step, count, M, prec):
    return dict(name=name, kind="batch", first=first, step=step, count=count, M=M, px=4, py=4, pz=2, pt=2, overlap=1,
                prec=prec, theta=0.5, faces=FACES, elem="q1", reg="h1h1")


def listed():
    return [
        # smallest call: the operator on a mesh of the parity tests (launch latency)
        _apply("apply64_small", (5, 4, 3), 6, 64, reg="h1l2"),
        # the outer operator of every solve, at the benchmark's size
        _apply("apply64_mid", (32, 32, 32), 64, 64),
        # the operator inside the mixed-precision preconditioner, at the paper's Example 1 and 2 mesh
        _apply("apply32_example", (40, 40, 40), 39, 32),
        # linear tetrahedra, an odd mesh
        _apply("apply64_p1", (27, 22, 25), 41, 64, elem="p1"),
        # the fine preconditioner of the benchmark: one apply per outer iteration
        _ras("ras32_mid", "ras", (32, 32, 32), 64, (4, 4, 4, 4), 2, 32),
        # the plain FP64 form, the batched workload's split, an odd mesh
        _ras("ras64_odd", "ras", (23, 19, 26), 37, (4, 4, 2, 2), 1, 64),
        # factors stored in 16 bits, the paper's examples (256 boxes, overlap 1)
        _ras("ras16_example", "ras", (40, 40, 40), 39, (4, 4, 4, 4), 1, 16),
        # exact local solves of the smallest workload (implicit Euler)
        _ras("ras_lu_tiny", "ras", (8, 8, 8), 16, (2, 2, 2, 2), 1, 64, local="lu", theta=1.0, faces=DIRICHLET_ALL),
        # the point-block ILU of the local-solver study (the paper's Table 1)
        _ras("ras_block", "ras", (16, 16, 16), 32, (4, 4, 4, 4), 1, 32, local="bilu0"),
        # new coefficients or regularisation: both levels refactored, then one two-level apply
        _ras("refactor_mid", "refactor", (32, 32, 32), 64, (4, 4, 4, 4), 2, 32),
        # the headline: observations to recovered source, two levels, mixed precision
        _ras("solve_mid", "solve", (32, 32, 32), 64, (4, 4, 4, 4), 2, 32),
        # several problems of uneven sizes solved together
        _batch("batch_solve", 16, 3, 3, 33, 32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "ras", "ras", "local", "refactor", "solve", "batch"])
    reg = rng.choice(["h1h1", "h1h1", "h1l2"])
    elem = rng.choice(["q1", "q1", "p1"])
    faces = rng.choice([1, 1, 9, 15])
    if kind == "apply":
        cells = [_log_int(rng, 3, 44) for _ in range(3)]
        return _unnamed(_apply("", cells, _log_int(rng, 4, 72), rng.choice([64, 64, 32]), elem, reg,
                               rng.choice([0.5, 0.5, 1.0]), faces))
    if kind == "ras":
        cells = [_log_int(rng, 7, 30) for _ in range(3)]
        split = rng.choice([(4, 4, 4, 4), (4, 4, 2, 2), (2, 2, 2, 2), (3, 2, 1, 4)])
        return _unnamed(_ras("", "ras", cells, _log_int(rng, 8, 56), split, rng.choice([0, 1, 1, 2]),
                             rng.choice([64, 32, 32, 16]), theta=rng.choice([0.5, 1.0]), faces=faces, elem=elem, reg=reg))
    if kind == "local":
        local = rng.choice(["bilu0", "bilu0", "ilu1", "lu"])
        if local == "lu":
            cells, M, split = [rng.randint(4, 8) for _ in range(3)], rng.randint(6, 16), (2, 2, 2, 2)
        elif local == "ilu1":
            cells, M, split = [rng.randint(4, 9) for _ in range(3)], rng.randint(5, 12), (3, 3, 3, 3)
        else:
            cells, M, split = [rng.randint(6, 16) for _ in range(3)], rng.randint(8, 32), rng.choice(
                [(4, 4, 4, 4), (4, 4, 2, 2)])
        return _unnamed(_ras("", "ras", cells, M, split, 1, 64 if local == "lu" else rng.choice([64, 32]), local=local,
                             faces=faces))
    if kind in ("refactor", "solve"):
        cells = [2 * _log_int(rng, 5, 13) for _ in range(3)]
        split = rng.choice([(4, 4, 4, 4), (4, 4, 2, 2), (2, 2, 2, 4)])
        return _unnamed(_ras("", kind, cells, 2 * _log_int(rng, 5, 24), split, rng.choice([1, 2]),
                             rng.choice([64, 32, 32]), elem=elem))
    return _unnamed(_batch("", rng.randint(8, 14), rng.randint(1, 3), rng.randint(2, 3), rng.randint(12, 33),
                           rng.choice([64, 32])))


def _unnamed(case):
    case.pop("name")
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _problem_data(case, seed, cells):
    """Coefficients, sensors and weights of one problem as numpy arrays (host)."""
    rng = np.random.default_rng([seed, 11, *cells, case["M"]])
    cx, cy, cz = cells
    ez, ey, ex = np.meshgrid(np.arange(cz), np.arange(cy), np.arange(cx), indexing="ij")
    xyz = np.stack([(ex.ravel() + 0.5) / cx, (ey.ravel() + 0.5) / cy, (ez.ravel() + 0.5) / cz], axis=1)
    rho = np.zeros(len(xyz))
    for _ in range(8):       # a smooth diffusivity between 0.05 and 0.1
        k = rng.integers(0, 4, 3)
        rho += rng.uniform(0.5, 1.0) * np.prod(np.cos(math.pi * k * xyz + rng.uniform(0, 2 * math.pi, 3)), axis=1)
    rho = (rho - rho.min()) / max(rho.max() - rho.min(), 1e-12)
    s = np.sin(math.pi * xyz[:, 2])
    v = np.stack([s, s, 0.1 * rng.uniform(-1, 1) * np.ones_like(s)], axis=1)
    m = 5 if min(cells) >= 12 else 3
    g = [np.round((np.arange(m) + 1.0) / (m + 1.0) * c).astype(int) for c in cells]
    z, y, x = np.meshgrid(g[2], g[1], g[0], indexing="ij")
    sens = (x + (cx + 1) * (y + (cy + 1) * z)).ravel().astype(np.int32)
    beta = 1e-3 * (32.0 / cx) ** 2
    return dict(cells=tuple(cells), a=0.05 + 0.05 * rho, v=v, sens=sens, beta1=beta / 100, beta2=beta,
                tau=1.0 / case["M"], m=m)


def _problem(case, d):
    p = api.Problem(d["cells"], LENGTHS, case["M"], d["tau"], d["a"], d["v"], d["sens"], d["beta1"], d["beta2"],
                    case["theta"], case["faces"])
    if case["reg"] != "h1h1":
        p.set_regularization(case["reg"])
    if case["elem"] != "q1":
        p.set_element(case["elem"])
    return p


def _random(n, seed, dtype=torch.float64):
    return torch.randn(n, dtype=dtype, device="cuda", generator=torch.Generator("cuda").manual_seed(seed + 1))


def _observations(case, d, seed):
    """Sensor signals of a cloud moving on a circle, with 1 % multiplicative noise."""
    rng = np.random.default_rng([seed, 12])
    t = np.arange(case["M"] + 1)[:, None] * d["tau"]
    nx, ny = d["cells"][0] + 1, d["cells"][1] + 1
    j = d["sens"].astype(np.int64)
    pos = np.stack([j % nx / d["cells"][0], j // nx % ny / d["cells"][1], j // (nx * ny) / d["cells"][2]], axis=1)
    ph = rng.uniform(0, 2 * math.pi)
    c = [0.5 + 0.25 * np.cos(2 * math.pi * t + ph), 0.5 + 0.25 * np.sin(2 * math.pi * t + ph), 0.55 + 0 * t]
    r2 = sum((pos[None, :, k] - c[k]) ** 2 for k in range(3))
    obs = 0.05 * t * np.exp(-r2 / 0.08) * (1 + 0.01 * rng.standard_normal(r2.shape))
    return torch.from_numpy(obs).cuda()


def _split(case):
    return (case["px"], case["py"], case["pz"], case["pt"])


def _cells(case):
    return (case["cx"], case["cy"], case["cz"])


def _batch_cells(case):
    return [(case["first"] + k * case["step"],) * 3 for k in range(case["count"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        data = [_problem_data(case, seed, c) for c in _batch_cells(case)]
        probs = [_problem(case, d) for d in data]
        ras = api.BatchRAS(probs, _split(case), case["overlap"], case["prec"])
        b = torch.cat([p.rhs(_observations(case, d, seed + k)) for k, (p, d) in enumerate(zip(probs, data))])
        return dict(kind=kind, probs=probs, ras=ras, b=b, x=torch.zeros_like(b))
    d = _problem_data(case, seed, _cells(case))
    p = _problem(case, d)
    if kind == "apply":
        x = _random(p.n, seed, torch.float64 if case["prec"] == 64 else torch.float32)
        return dict(kind=kind, prob=p, x=x, y=torch.empty_like(x))
    state = dict(kind=kind, prob=p)
    state["ras"] = api.RAS(p, _split(case), case["overlap"], case["prec"], local=case["local"])
    if kind != "ras":
        state["coarse"] = api.Coarse(p, tuple(c // 2 for c in _cells(case)), case["M"] // 2, _split(case),
                                     factor_prec=case["prec"])
    if kind == "solve":
        state["obs"] = _observations(case, d, seed)
        state["b"], state["x"] = p.zeros(), p.zeros()
    else:
        state["r"] = _random(p.n, seed)
        state["z"] = torch.empty_like(state["r"])
    return state


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return state["prob"].apply(state["x"], out=state["y"])
    if kind == "ras":
        return state["ras"].apply(state["r"], out=state["z"])
    if kind == "refactor":
        state["coarse"].refactor_with(state["ras"])
        return state["coarse"].apply(state["ras"], state["r"], out=state["z"])
    state["x"].zero_()
    if kind == "batch":
        x, _, _, its, _ = api.gmres_solve_batch(state["probs"], state["ras"], state["b"], state["x"])
        return dict(x=x, iterations=its)
    p = state["prob"]
    p.rhs(state["obs"], out=state["b"])
    state["coarse"].refactor_with(state["ras"])
    x, _, its, _ = api.gmres_solve(p, state["b"], state["x"], ras=state["ras"], coarse=state["coarse"])
    return dict(x=x, source=p.recover_source(x), iterations=its)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _box_points(cells, M, split, overlap):
    total = 1
    for n, p in zip((*(c + 1 for c in cells), M + 1), split):
        total *= sum(hi - lo for lo, hi in _parts(n, p, overlap)[0])
    return total


def _parts(n, p, overlap):
    """Extended and owned ranges of the p parts of n points."""
    own, s = [], 0
    for k in range(p):
        e = s + n // p + (k < n % p)
        own.append((s, e))
        s = e
    return [(max(0, a - overlap), min(n, b + overlap)) for a, b in own], own


def _matvec_work(cells, M, prec, elem):
    nodes = math.prod(c + 1 for c in cells)
    points = nodes * (M + 1)
    esz = 4 if prec == 32 else 8
    coef = 2 * 27 if elem == "q1" else 4 * 15
    return points * 6 * esz + nodes * coef * esz, points * (230 if elem == "q1" else 220)


def _local_work(case, cells, M):
    """Bytes and flops of one RAS apply, and values per box point."""
    points = math.prod(c + 1 for c in cells) * (M + 1)
    box = _box_points(cells, M, _split(case), case["overlap"])
    if case.get("local") == "lu":
        n = [hi - lo for lo, hi in _parts(cells[0] + 1, case["px"], case["overlap"])[0]][0]
        values = 3 * 3 * 3 * (1 + n + n * n + n ** 3)      # a band of L and U with row interchanges
    else:
        values = {"ilu1": 1646, "bilu0": 729}.get(case.get("local"), 326)
    return box * (values * VALUE_BYTES[case["prec"]] + 24) + 24 * points, 2.0 * box * values


def work(case):
    kind, M = case["kind"], case["M"]
    if kind == "apply":
        nbytes, flops = _matvec_work(_cells(case), M, case["prec"], case["elem"])
        return dict(bytes=nbytes, flops=flops)
    if kind == "ras":
        nbytes, flops = _local_work(case, _cells(case), M)
        return dict(bytes=nbytes, flops=flops)
    nbytes = flops = 0.0
    esz = VALUE_BYTES[case["prec"]]
    if kind == "batch":
        for cells in _batch_cells(case):
            mb, mf = _matvec_work(cells, M, 64, "q1")
            lb, lf = _local_work(case, cells, M)
            nbytes += 3 * ITERATIONS * (mb + lb)
            flops += 3 * ITERATIONS * (mf + lf)
        return dict(bytes=nbytes, flops=flops)
    applies = 1 if kind == "refactor" else ITERATIONS
    coarse = tuple(c // 2 for c in _cells(case))
    for cells, m, overlap, reps in ((_cells(case), M, case["overlap"], applies), (coarse, M // 2, 1, 4 * applies)):
        box = _box_points(cells, m, _split(case), overlap)
        lb, lf = _local_work(dict(case, overlap=overlap), cells, m)
        mb, mf = _matvec_work(cells, m, 32 if case["prec"] != 64 else 64, case["elem"])
        nbytes += 2 * 326 * esz * box + reps * (lb + mb)
        flops += 2 * 3739.0 * box + reps * (lf + mf)
    if kind == "solve":
        mb, mf = _matvec_work(_cells(case), M, 64, case["elem"])
        points = math.prod(c + 1 for c in _cells(case)) * (M + 1)
        nbytes += applies * (mb + 24 * points * (ITERATIONS + 3))
        flops += applies * mf
    return dict(bytes=nbytes, flops=flops)


# ---------------------------------------------------------------------------
# the same in 64 bits, with plain torch
# ---------------------------------------------------------------------------

def _cell_matrices(h, elem):
    """Mass, stiffness and the three convection matrices (test a, trial b) of one cell, 8 nodes x fastest."""
    hx = np.asarray(h)
    corner = np.array([[(a >> k) & 1 for k in range(3)] for a in range(8)], dtype=float)
    B, K, E = np.zeros((8, 8)), np.zeros((8, 8)), np.zeros((3, 8, 8))
    if elem == "q1":
        g = 0.5 + np.array([-0.5, 0.5]) / math.sqrt(3.0)
        for px in g:
            for py in g:
                for pz in g:
                    x = np.array([px, py, pz])
                    f = np.where(corner == 1, x, 1 - x)                      # (8, 3) one-dimensional factors
                    N = f.prod(axis=1)
                    D = np.stack([np.where(corner[:, k] == 1, 1.0, -1.0) / hx[k] *
                                  np.delete(f, k, axis=1).prod(axis=1) for k in range(3)])
                    w = hx.prod() / 8
                    B += w * np.outer(N, N)
                    K += w * sum(np.outer(D[k], D[k]) for k in range(3))
                    E += w * np.stack([np.outer(N, D[k]) for k in range(3)])
        return B, K, E
    # six tetrahedra around the main diagonal: one for each order of the axes
    for axes in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        nodes = [0]
        for k in axes:
            nodes.append(nodes[-1] | (1 << k))
        X = np.concatenate([np.ones((4, 1)), corner[nodes] * hx], axis=1)
        grad = np.linalg.inv(X)[1:]                                          # (3, 4)
        vol = hx.prod() / 6
        ix = np.ix_(nodes, nodes)
        B[ix] += vol / 20 * (np.ones((4, 4)) + np.eye(4))
        K[ix] += vol * grad.T @ grad
        for k in range(3):
            E[k][ix] += vol / 4 * np.outer(np.ones(4), grad[k])
    return B, K, E


class _Exact:
    """F_h of one problem in 64 bits: 27-point row stencils of B, K, S = A + E and S^T."""

    def __init__(self, case, d):
        cx, cy, cz = self.cells = d["cells"]
        self.shape = (cz + 1, cy + 1, cx + 1)
        self.N, self.M, self.L = math.prod(self.shape), case["M"], case["M"] + 1
        self.tau, self.theta, self.reg = d["tau"], case["theta"], case["reg"]
        self.beta1, self.beta2 = d["beta1"], d["beta2"]
        Bc, Kc, Ec = _cell_matrices([1.0 / c for c in self.cells], case["elem"])
        a = torch.from_numpy(d["a"]).reshape(cz, cy, cx).cuda()
        v = torch.from_numpy(d["v"]).reshape(cz, cy, cx, 3).cuda()
        self.B, self.K, self.S, self.ST = (torch.zeros(27, *self.shape, dtype=torch.float64, device="cuda")
                                           for _ in range(4))
        for i in range(8):
            for j in range(8):
                o = [((j >> k) & 1) - ((i >> k) & 1) + 1 for k in range(3)]
                q = o[0] + 3 * o[1] + 9 * o[2]
                row = tuple(slice((i >> k) & 1, ((i >> k) & 1) + n) for k, n in ((2, cz), (1, cy), (0, cx)))
                self.B[q][row] += Bc[i, j]
                self.K[q][row] += Kc[i, j]
                self.S[q][row] += a * Kc[i, j] + sum(v[..., k] * Ec[k, i, j] for k in range(3))
                self.ST[q][row] += a * Kc[i, j] + sum(v[..., k] * Ec[k, j, i] for k in range(3))
        dirichlet = torch.zeros(self.shape, dtype=torch.bool, device="cuda")
        for face, at in enumerate(((slice(None), slice(None), 0), (slice(None), slice(None), -1),
                                   (slice(None), 0), (slice(None), -1), (0,), (-1,))):
            if case["faces"] >> face & 1:
                dirichlet[at] = True
        self.dirichlet = dirichlet
        sens = torch.zeros(self.N, dtype=torch.float64, device="cuda")
        sens.index_add_(0, torch.from_numpy(d["sens"].astype(np.int64)).cuda(),
                        torch.ones(len(d["sens"]), dtype=torch.float64, device="cuda"))
        self.sens = sens.reshape(self.shape) * ~dirichlet
        n = torch.arange(self.L, device="cuda", dtype=torch.float64)
        sides = ((n > 0).double() + (n < self.M).double())
        self.mt0, self.lt0 = self.tau / 3 * sides, sides / self.tau
        self.mt1, self.lt1 = self.tau / 6, -1.0 / self.tau

    def stencil(self, coef, u):
        nz, ny, nx = self.shape
        up = torch.nn.functional.pad(u, (1, 1, 1, 1, 1, 1))
        out = torch.zeros_like(u)
        for q in range(27):
            x, y, z = q % 3, q // 3 % 3, q // 9
            out += coef[q] * up[:, z:z + nz, y:y + ny, x:x + nx]
        return out

    def apply(self, x):
        C, G, f = (x.reshape(self.L, *self.shape, 3)[..., k].contiguous() for k in range(3))
        zero = torch.zeros_like(C[:1])
        before = lambda u: torch.cat([zero, u[:-1]])                         # noqa: E731
        after = lambda u: torch.cat([u[1:], zero])                           # noqa: E731
        lv = lambda w: w.reshape(-1, 1, 1, 1)                                # noqa: E731
        th, th1, tau = self.theta, 1 - self.theta, self.tau
        yC = self.stencil(self.B, C - before(C) - tau * (th * f + th1 * before(f))) + \
            tau * self.stencil(self.S, th * C + th1 * before(C))
        yG = self.stencil(self.B, G - after(G)) + tau * self.stencil(self.ST, th * G + th1 * after(G)) + \
            tau * self.sens * (th * after(C) + th1 * C)
        Mt = lambda u: lv(self.mt0) * u + self.mt1 * (before(u) + after(u))  # noqa: E731
        Lt = lambda u: lv(self.lt0) * u + self.lt1 * (before(u) + after(u))  # noqa: E731
        yf = self.stencil(self.B, self.beta1 * Lt(f) - Mt(G)) + \
            self.beta2 * self.stencil(self.K if self.reg == "h1h1" else self.B, Mt(f))
        yC[0], yG[-1] = C[0], G[-1]
        yC, yG = torch.where(self.dirichlet, C, yC), torch.where(self.dirichlet, G, yG)
        return torch.stack([yC, yG, yf], dim=-1).reshape(-1)

    def entries(self, c, dt, q, cc, node, level):
        """Values of the column (level + dt, node + offset q, component cc) in rows (level, node, c)."""
        th, th1, tau = self.theta, 1 - self.theta, self.tau
        at = lambda coef: coef.reshape(27, -1)[q][node]                      # noqa: E731
        zero = torch.zeros(node.shape, dtype=torch.float64, device="cuda")
        fixed = self.dirichlet.reshape(-1)[node]
        diagonal = c == cc and dt == 0 and q == 13
        if c == 0:
            fixed = fixed | (level == 0)
            val = zero
            if cc == 0 and dt <= 0:
                val = at(self.B) * (1 if dt == 0 else -1) + (th if dt == 0 else th1) * tau * at(self.S)
            elif cc == 2 and dt <= 0:
                val = -(th if dt == 0 else th1) * tau * at(self.B)
        elif c == 1:
            fixed = fixed | (level == self.M)
            val = zero
            if cc == 1 and dt >= 0:
                val = at(self.B) * (1 if dt == 0 else -1) + (th if dt == 0 else th1) * tau * at(self.ST)
            elif cc == 0 and dt >= 0 and q == 13:
                val = (th1 if dt == 0 else th) * tau * self.sens.reshape(-1)[node]
        else:
            if cc == 0:
                return zero
            mt = self.mt0[level] if dt == 0 else self.mt1
            lt = self.lt0[level] if dt == 0 else self.lt1
            if cc == 1:
                return -mt * at(self.B)
            return self.beta1 * lt * at(self.B) + self.beta2 * mt * at(self.K if self.reg == "h1h1" else self.B)
        return torch.where(fixed, torch.full_like(val, 1.0 if diagonal else 0.0), val)


def _slots(c, blocks):
    """Columns of row type c in column order: (offset in the 81-point neighbourhood, component)."""
    out = []
    for dt in (-1, 0, 1):
        for q in range(27):
            for cc in range(3):
                if blocks or (c == 0 and dt <= 0 and cc != 1) or (c == 2 and cc != 0) or \
                        (c == 1 and dt >= 0 and (cc == 1 or (cc == 0 and q == 13))):
                    out.append((27 * (dt + 1) + q, cc))
    return out


def _vector(o):
    return np.array([o % 3 - 1, o // 3 % 3 - 1, o // 9 % 3 - 1, o // 27 - 1])


class _Boxes:
    """The points of all extended boxes of a split, and their 81 neighbours within their box."""

    def __init__(self, F, split, overlap):
        dims = (F.shape[2], F.shape[1], F.shape[0], F.L)
        ext, own = zip(*(_parts(n, p, overlap) for n, p in zip(dims, split)))
        node, level, wave, nbr, owned, self.sizes = [], [], [], [], [], []
        base = 0
        for kt in range(split[3]):
            for kz in range(split[2]):
                for ky in range(split[1]):
                    for kx in range(split[0]):
                        lo = [ext[a][k][0] for a, k in enumerate((kx, ky, kz, kt))]
                        hi = [ext[a][k][1] for a, k in enumerate((kx, ky, kz, kt))]
                        l = [h - b for b, h in zip(lo, hi)]
                        t, z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda") for n in l[::-1]), indexing="ij")
                        local = [x.reshape(-1), y.reshape(-1), z.reshape(-1), t.reshape(-1)]
                        node.append(local[0] + lo[0] + dims[0] * (local[1] + lo[1] + dims[1] * (local[2] + lo[2])))
                        level.append(local[3] + lo[3])
                        wave.append(local[0] + 2 * local[1] + 4 * local[2] + 8 * local[3])
                        inside = torch.ones_like(local[0], dtype=torch.bool)
                        for a, k in enumerate((kx, ky, kz, kt)):
                            g = local[a] + lo[a]
                            inside &= (g >= own[a][k][0]) & (g < own[a][k][1])
                        owned.append(inside)
                        lex = torch.arange(len(inside), device="cuda")
                        table = torch.full((len(inside), 81), -1, dtype=torch.int32, device="cuda")
                        for o in range(81):
                            v = _vector(o)
                            ok = torch.ones_like(inside)
                            for a in range(4):
                                ok &= (local[a] + int(v[a]) >= 0) & (local[a] + int(v[a]) < l[a])
                            step = int(v[0] + l[0] * (v[1] + l[1] * (v[2] + l[2] * v[3])))
                            table[:, o] = torch.where(ok, lex + step + base, -1).int()
                        nbr.append(table)
                        self.sizes.append(len(lex))
                        base += len(lex)
        self.P = base
        self.node, self.level, self.owned = torch.cat(node), torch.cat(level), torch.cat(owned)
        self.nbr = torch.cat(nbr)
        self.nbr[self.nbr < 0] = base                                        # outside: the spare point
        wave = torch.cat(wave)
        order = torch.argsort(wave, stable=True)
        ends = torch.cumsum(torch.bincount(wave), 0).tolist()
        self.waves = [order[a:b] for a, b in zip([0] + ends[:-1], ends)]
        self.unknown = 3 * (self.level * F.N + self.node)


def _exact_ilu(F, boxes, r, blocks):
    """One-level RAS apply with ILU(0) (scalar, or on whole point blocks), in 64 bits."""
    rows = [_slots(c, blocks) for c in range(3)]
    base = [0, len(rows[0]), len(rows[0]) + len(rows[1])]
    where = {(c, o, cc): k for c in range(3) for k, (o, cc) in enumerate(rows[c])}
    diag = [where[c, 40, c] for c in range(3)]
    A = torch.zeros(boxes.P + 1, sum(map(len, rows)), dtype=torch.float64, device="cuda")
    for c in range(3):
        for k, (o, cc) in enumerate(rows[c]):
            val = F.entries(c, o // 27 - 1, o % 27, cc, boxes.node, boxes.level)
            A[:-1, base[c] + k] = val * (boxes.nbr[:, o] < boxes.P)
        A[-1, base[c] + diag[c]] = 1.0                                       # reciprocal pivots on the diagonals
    plan = []
    for c in range(3):
        for s, (o, cc) in enumerate(rows[c][:diag[c]]):
            pairs = []
            for t in range(diag[cc] + 1, len(rows[cc])):
                v = _vector(o) + _vector(rows[cc][t][0])
                if np.abs(v).max() <= 1:
                    u = where.get((c, int((v + 1) @ [1, 3, 9, 27]), rows[cc][t][1]))
                    if u is not None:
                        pairs.append((base[cc] + t, u))
            t, u = (torch.tensor(list(z), device="cuda", dtype=torch.int64) for z in (zip(*pairs) if pairs else ((), ())))
            plan.append((c, s, o, base[cc] + diag[cc], t, u))
    spans = [slice(base[c], base[c] + len(rows[c])) for c in range(3)]
    for p in boxes.waves:
        nb = boxes.nbr[p].long()
        for c in range(3):
            R = A[p, spans[c]]
            for (k, s, o, d, t, u) in plan:
                if k != c:
                    continue
                q = nb[:, o]
                R[:, s] *= A[q, d]
                if len(t):
                    R.index_add_(1, u, R[:, s:s + 1] * A[q[:, None], t], alpha=-1)
            R[:, diag[c]] = 1.0 / R[:, diag[c]]
            A[p, spans[c]] = R
    V = torch.zeros(boxes.P + 1, 3, dtype=torch.float64, device="cuda")
    V[:-1] = r[boxes.unknown[:, None] + torch.arange(3, device="cuda")]
    off = [torch.tensor([o for o, _ in rows[c]], device="cuda") for c in range(3)]
    comp = [torch.tensor([cc for _, cc in rows[c]], device="cuda") for c in range(3)]
    for lower in (True, False):
        for p in boxes.waves if lower else boxes.waves[::-1]:
            nb = boxes.nbr[p].long()
            for c in (0, 1, 2) if lower else (2, 1, 0):
                part = slice(0, diag[c]) if lower else slice(diag[c] + 1, len(rows[c]))
                acc = V[p, c] - (A[p, spans[c]][:, part] * V[nb[:, off[c][part]], comp[c][part]]).sum(1)
                V[p, c] = acc if lower else acc * A[p, base[c] + diag[c]]
    return _owned(boxes, V[:-1], r)


def _exact_lu(F, boxes, r):
    """One-level RAS apply with exact local solves, in 64 bits."""
    V = torch.zeros(boxes.P, 3, dtype=torch.float64, device="cuda")
    start = 0
    for size in boxes.sizes:
        sl = slice(start, start + size)
        A = torch.zeros(3 * size, 3 * size, dtype=torch.float64, device="cuda")
        row = 3 * torch.arange(size, device="cuda")
        for c in range(3):
            for (o, cc) in _slots(c, False):
                col = boxes.nbr[sl, o].long()
                ok = col < boxes.P
                val = F.entries(c, o // 27 - 1, o % 27, cc, boxes.node[sl], boxes.level[sl])
                A[row[ok] + c, 3 * (col[ok] - start) + cc] = val[ok]
        rhs = r[boxes.unknown[sl][:, None] + torch.arange(3, device="cuda")].reshape(-1, 1)
        V[sl] = torch.linalg.solve(A, rhs).reshape(-1, 3)
        start += size
    return _owned(boxes, V, r)


def _owned(boxes, V, r):
    z = torch.zeros_like(r)
    z[boxes.unknown[boxes.owned][:, None] + torch.arange(3, device="cuda")] = V[boxes.owned]
    return z


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("apply", "ras") or case.get("local") == "ilu1":
        return None          # iterative, or a pattern that grows by fill
    d = _problem_data(case, seed, _cells(case))
    F = _Exact(case, d)
    n = 3 * F.N * F.L
    if kind == "apply":
        return F.apply(_random(n, seed, torch.float64 if case["prec"] == 64 else torch.float32).double())
    boxes = _Boxes(F, _split(case), case["overlap"])
    if case["local"] == "lu":
        return _exact_lu(F, boxes, _random(n, seed))
    return _exact_ilu(F, boxes, _random(n, seed), case["local"] == "bilu0")
