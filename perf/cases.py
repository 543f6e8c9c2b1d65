"""The work a user of this library has it do, as measurable cases.

A case is one call (or one round of requests) through the public Python
binding on a problem that the program keeps set up: a preconditioner apply, a
PCG solve on device or host vectors, an interface-reduced solve, a round of
served requests, or the setup for a new coefficient followed by its solve.

The problems are those of ``inputs.py`` (its generators, at the sizes of the
configurations, tests and benchmark and between them).  Solves run to a
relative residual of 1e-10, the tighter of the two tolerances the tests use:
there the solution is determined by the problem to many more digits than by
the iterates that led to it.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_0911_5730_gb300 import bddc, inputs

RTOL = 1e-10
MAXIT = 1000


# --------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------
def _case(name, problem, nx, kind, precision, nrhs):
    c = {"problem": problem, "nx": nx, "kind": kind, "precision": precision, "nrhs": nrhs}
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest problem of the configurations: one right-hand side, all
        # launch latency (a coarse model, an inner solve, a unit test)
        _case("unit_32_fp64_1", "unit", 32, "solve", "fp64", 1),
        # the benchmark's problem, one right-hand side at a time, as an
        # interactive client or a time step sees it
        _case("channels_512_fp32_1", "channels", 512, "solve", "fp32", 1),
        # one FP64 preconditioner application inside a user's own Krylov loop
        _case("channels_512_apply_fp64_1", "channels", 512, "apply", "fp64", 1),
        # the FP64 solve of one right-hand side in the form that is the fastest
        # there (level 1 reduced to its interface)
        _case("channels_512_reduced_fp64_1", "channels", 512, "reduced", "fp64", 1),
        # the benchmark's step end to end: 96 right-hand sides from and to
        # pinned host buffers
        _case("channels_512_host_fp32_96", "channels", 512, "host", "fp32", 96),
        # a full batch with the FP64 apply
        _case("channels_512_fp64_32", "channels", 512, "solve", "fp64", 32),
        # a round of served requests of 1 to 64 right-hand sides
        _case("channels_256_serve_fp32_87", "channels", 256, "serve", "fp32", 87),
        # three levels, a million unknowns: one right-hand side, and a batch
        _case("blocks_1024_fp32_1", "blocks", 1024, "solve", "fp32", 1),
        _case("blocks_1024_fp32_32", "blocks", 1024, "solve", "fp32", 32),
        # irregular substructures, a batch that fills no group
        _case("voronoi_1024_fp32_21", "voronoi", 1024, "solve", "fp32", 21),
        # plane elasticity on three levels with the jagged edges
        _case("elasticity_384_fp32_1", "elasticity", 384, "solve", "fp32", 1),
        # a new coefficient field: setup, selection and one solve
        _case("channels_512_setup_fp32_1", "channels", 512, "setup", "fp32", 1),
    ]


#: sizes each problem is drawn at: (step of nx, smallest, largest)
_SIZES = {"unit": (8, 32, 512), "channels": (16, 64, 512), "blocks": (64, 128, 1024),
          "voronoi": (128, 256, 1024), "elasticity": (48, 96, 384)}


def _cost(c):
    """A rough cost of a case, to keep drawn ones below the largest listed one."""
    w = work(c)
    return w["flops"] * (8.0 if c["precision"] == "fp64" else 1.0)


def draw(rng):
    top = max(_cost(c) for c in listed())
    while True:
        problem = rng.choice(["unit", "channels", "channels", "blocks", "voronoi", "elasticity"])
        step, lo, hi = _SIZES[problem]
        nx = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step
        nx = min(max(nx, lo), hi)
        kind = rng.choice(["solve", "solve", "solve", "apply", "host", "serve", "reduced", "setup"])
        precision = rng.choice(["fp32", "fp32", "fp64"])
        nrhs = 1 if rng.random() < 0.35 else int(round(math.exp(rng.uniform(math.log(2), math.log(96)))))
        if kind in ("reduced", "setup"):
            nrhs = 1
        if kind == "apply":
            precision = "fp64"
        if problem == "elasticity" and nrhs > 8:
            nrhs = 1 + nrhs % 8     # levels beyond the batch kernels: a loop over right-hand sides
        c = _case(None, problem, nx, kind, precision, nrhs)
        if _cost(c) <= top:
            return c


# --------------------------------------------------------------------------
# problems
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _voronoi(nx):
    """The cells of a size (the mesh a program keeps; its coefficient varies)."""
    cells = nx // 32
    return inputs.voronoi_decomposition(nx, cells, 4001, 0.25, 8 if cells % 8 == 0 and cells > 8 else 4)


def _workload(problem, nx, seed):
    if problem == "unit":           # k = 1, corners + edge averages, 8 x 8-element substructures
        return inputs.two_level_unit(nx, 8)
    if problem == "channels":       # 1e6 channels, adaptive tau = 10, 16 x 16-element substructures
        return inputs.two_level_channels(nx, 16, 10.0, seed=2001 + seed)
    if problem == "blocks":         # log10 k in [0, 6] per 8 x 8 block, three levels
        return inputs.three_level_blocks(nx, 8, 8, 10.0, seed=3001 + seed)
    if problem == "voronoi":        # cells of about 1000 elements, three levels
        e2s, ns, s2, n2 = _voronoi(nx)
        return inputs.Workload("voronoi_%d" % nx, nx, inputs.block_log_uniform_coefficient(nx, 8, 4002 + seed),
                               e2s, ns, 3, 10.0, "adaptive", s2, n2)
    # plane elasticity: three levels, 3 x 3 level-2 substructures, Lame
    # parameters within a factor of two of each other
    m = nx // 16
    k = 2.0 ** np.random.default_rng(71 + seed).uniform(0.0, 1.0, nx * nx)
    return inputs.elasticity(nx, 16, 3, m // 3, "adaptive", 3.0, jagged=m // 3 >= 8, k=k)


def _seed(seed):
    return int(seed) % (1 << 31)


def _rhs(n, nrhs, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(_seed(seed))
    shape = (n,) if nrhs == 1 else (nrhs, n)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)


def _requests(nrhs):
    """A round of requests: sizes 1, 2, 4, ... up to 64, the last cut to what is left."""
    sizes, left, s = [], nrhs, 1
    while left:
        sizes.append(min(s, left))
        left -= sizes[-1]
        s = 1 if s == 64 else 2 * s
    return sizes


def prepare(case, seed):
    wl = _workload(case["problem"], case["nx"], _seed(seed))
    n, nrhs, kind = wl.n_dof, case["nrhs"], case["kind"]
    b = _rhs(n, nrhs, seed)
    if kind == "setup":
        return {"kind": kind, "wl": wl, "precision": case["precision"], "b": b}
    if kind == "serve":
        st = {"kind": kind, "srv": bddc.Server(), "prob": bddc.Problem.from_workload(wl, precision=case["precision"])}
        rows = b.cpu().numpy().reshape(nrhs, n)
        ends = np.cumsum(_requests(nrhs))
        st["reqs"] = [np.ascontiguousarray(rows[e - s:e]) for s, e in zip(_requests(nrhs), ends)]
        return st
    st = {"kind": kind, "prob": bddc.Problem.from_workload(wl, precision=case["precision"])}
    if kind == "host":
        st["b"] = b.cpu().pin_memory()
        st["x"] = torch.empty_like(st["b"]).pin_memory()
    else:
        st["b"] = b
    return st


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return state["prob"].apply(state["b"])
    if kind == "solve":
        return state["prob"].solve(state["b"], rtol=RTOL, maxit=MAXIT)[0]
    if kind == "reduced":
        return state["prob"].solve_reduced(state["b"], rtol=RTOL, maxit=MAXIT)[0]
    if kind == "host":
        return state["prob"].solve_host(state["b"], state["x"], rtol=RTOL, maxit=MAXIT)[0]
    if kind == "serve":
        srv, prob = state["srv"], state["prob"]
        tickets = [srv.submit(prob, b, rtol=RTOL, maxit=MAXIT) for b in state["reqs"]]
        return [srv.wait(t)[0] for t in tickets]
    # setup: a new coefficient, the selected constraints and the solution
    prob = bddc.Problem.from_workload(state["wl"], precision=state["precision"])
    x = prob.solve(state["b"], rtol=RTOL, maxit=MAXIT)[0]
    q = prob.query(level=1)
    prob.close()
    return {"x": x, "eigs": q["edge_eigs"], "selected": q["n_selected"]}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
#: PCG iterations to RTOL, about
_ITERS = {"unit": 9, "channels": 33, "blocks": 45, "voronoi": 47, "elasticity": 17}


def work(case):
    """Vectors in and out once, the operators (banded interior factors, dense
    interface operators, stencil) once in the precision of the apply; the
    multiply-adds of the sweeps (two interior solves of two sweeps), the
    interface operator, the stencil and the recurrences, per iteration."""
    problem, nx, nrhs = case["problem"], case["nx"], case["nrhs"]
    el = problem == "elasticity"
    n = 2 * nx * (nx + 1) if el else (nx - 1) ** 2
    side = {"unit": 8, "channels": 16, "blocks": 8, "voronoi": 32, "elasticity": 16}[problem]
    dofs = 2 if el else 1
    band = dofs * (side + 1)                         # half bandwidth of an interior
    sub = (nx / side) ** 2                           # substructures
    n_gamma = dofs * 4 * side                        # interface DOFs of one
    factor, dense = n * band, sub * n_gamma ** 2
    e = 8 if case["precision"] == "fp64" else 4
    its = 1 if case["kind"] == "apply" else _ITERS[problem]
    sweeps = 2 if case["kind"] == "reduced" else 4
    fma = nrhs * (sweeps * factor + dense + n * ((46 if el else 9) + 6)) * its
    out = {"bytes": 16.0 * n * nrhs + e * (factor + dense) + 40.0 * n, "flops": 2.0 * fma}
    if case["kind"] == "setup":                      # factorisation, Schur complements, inverses
        out["flops"] += 2.0 * (n * band * (band / 2 + n_gamma) + sub * n_gamma ** 3)
    return out


# --------------------------------------------------------------------------
# the same in 64 bits: a direct solve, block elimination over the mesh rows
# --------------------------------------------------------------------------
def _rows_diffusion(nx, k):
    """Diagonal and lower off-diagonal blocks (dense rows of the mesh) of the
    Q1 operator with zero boundary values: functions of the row."""
    k = torch.as_tensor(np.ascontiguousarray(k), device="cuda").reshape(nx, nx)     # [ej, ei]
    s, n_ = k[:-1], k[1:]                                       # elements below and above each node row
    sw, se, nw, ne = s[:, :-1], s[:, 1:], n_[:, :-1], n_[:, 1:]
    dia = (sw + se + nw + ne) * (4.0 / 6.0)                     # [node row, node column]
    east = -(se + ne)[:, :-1] / 6.0
    north = -(ne + nw) / 6.0
    north_e, north_w = -2.0 * ne[:, :-1] / 6.0, -2.0 * nw[:, 1:] / 6.0

    def diag(j):
        return torch.diag(dia[j]) + torch.diag(east[j], 1) + torch.diag(east[j], -1)

    def low(j):     # A[row j + 1, row j]: node (i, j + 1) sees (i, j) and its neighbours
        # node (i, j) couples to (i + 1, j + 1) by its NE element, to (i - 1, j + 1) by its NW element
        return torch.diag(north[j]) + torch.diag(north_e[j], -1) + torch.diag(north_w[j], 1)

    return nx - 1, diag, low


def _rows_elasticity(nx, k, lame):
    """The same for plane strain with bilinear elements, clamped on x = 0;
    a node row holds nodes 1..nx with two components each."""
    lam, mu = lame
    g = 1.0 / math.sqrt(3.0)
    d = np.array([[lam + 2 * mu, lam, 0.0], [lam, lam + 2 * mu, 0.0], [0.0, 0.0, mu]])
    ke = np.zeros((8, 8))
    xs, ys = np.array([-1.0, 1.0, 1.0, -1.0]), np.array([-1.0, -1.0, 1.0, 1.0])
    for a in (-g, g):
        for c in (-g, g):
            dx, dy = xs * (1 + ys * c) / 4, ys * (1 + xs * a) / 4       # reference derivatives
            bm = np.zeros((3, 8))
            bm[0, 0::2], bm[1, 1::2] = dx, dy
            bm[2, 0::2], bm[2, 1::2] = dy, dx
            ke += bm.T @ d @ bm                # the map's factors cancel for square elements
    ke = torch.as_tensor(ke, device="cuda")
    k = torch.as_tensor(np.ascontiguousarray(k), device="cuda").reshape(nx, nx)
    loc = {(0, 0): 0, (1, 0): 1, (1, 1): 2, (0, 1): 3}                  # (right, upper) -> local node
    ei = torch.arange(nx, device="cuda")

    def add(m, ej, up_r, up_c):
        """The couplings of element row ej between its lower/upper node rows."""
        for rr in (0, 1):
            for cc in (0, 1):
                blk = ke[2 * loc[rr, up_r]:2 * loc[rr, up_r] + 2, 2 * loc[cc, up_c]:2 * loc[cc, up_c] + 2]
                r, c = ei + rr - 1, ei + cc - 1                         # column index among nodes 1..nx
                ok = (r >= 0) & (c >= 0)
                for p in (0, 1):
                    for q in (0, 1):
                        m.index_put_((2 * r[ok] + p, 2 * c[ok] + q), k[ej][ok] * blk[p, q], accumulate=True)
        return m

    def zero():
        return torch.zeros(2 * nx, 2 * nx, dtype=torch.float64, device="cuda")

    def diag(j):
        m = zero()
        if j > 0:
            add(m, j - 1, 1, 1)
        if j < nx:
            add(m, j, 0, 0)
        return m

    def low(j):
        return add(zero(), j, 1, 0)

    return nx + 1, diag, low


def _direct(rows, b):
    """x with A x = b, A block tridiagonal; b [nrhs, n] on the GPU."""
    m, diag, low = rows
    w = b.shape[1] // m
    rhs = b.reshape(b.shape[0], m, w).permute(1, 2, 0).contiguous()     # [row, w, nrhs]
    chol, y = [], []
    for j in range(m):
        s, v = diag(j), rhs[j]
        if j > 0:
            e = low(j - 1)
            s = s - e @ torch.cholesky_solve(e.T.contiguous(), chol[-1])
            v = v - e @ torch.cholesky_solve(y[-1], chol[-1])
        chol.append(torch.linalg.cholesky((s + s.T) / 2))
        y.append(v)
    x = [None] * m
    for j in range(m - 1, -1, -1):
        v = y[j] if j == m - 1 else y[j] - low(j).T @ x[j + 1]
        x[j] = torch.cholesky_solve(v, chol[j])
    return torch.stack(x).permute(2, 0, 1).reshape(b.shape)


def exact(case, seed):
    if case["kind"] == "apply":          # the preconditioner itself: no closed form without its construction
        return None
    wl = _workload(case["problem"], case["nx"], _seed(seed))
    b = _rhs(wl.n_dof, case["nrhs"], seed)
    if case["problem"] == "elasticity":
        rows = _rows_elasticity(wl.nx, wl.k, wl.lame)
    else:
        rows = _rows_diffusion(wl.nx, wl.k)
    x = _direct(rows, b.reshape(-1, wl.n_dof)).reshape(b.shape)
    if case["kind"] == "serve":
        ends = np.cumsum(_requests(case["nrhs"]))
        xs = [x.reshape(case["nrhs"], -1)[e - s:e].cpu().numpy() for s, e in zip(_requests(case["nrhs"]), ends)]
        return [v.reshape(-1) if v.shape[0] == 1 else v for v in xs]
    if case["kind"] == "setup":
        return {"x": x, "eigs": None, "selected": None}
    return x.cpu() if case["kind"] == "host" else x
