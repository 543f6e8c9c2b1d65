"""The kernels at the sizes where their tiles, rings and dispatch rules turn:
right-hand-side counts on both sides of each rule and ragged against the
copy tiles, blocks whose off-diagonal factor is triangular and ones where it
is not, block sizes on both sides of the factorisation's shared memory, and
substructures too large for the one-record-per-lane kernels.

The reference is the CPU oracle (or, at sizes that take it long, the FP64
apply of the same problem, which the other files compare with the oracle);
the tolerances are the parity ones: 1e-10 for FP64 applies, 1e-5 for FP32
applies, a true relative residual of 1e-8.  BF16 applies, iteration counts and
solution errors are compared in the other files: here the coefficient jumps of
1e6 leave more than their tolerances to the rounding of the operators and to
the stopping test.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import bddc as obddc          # noqa: E402
from paper_0911_5730_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0911_5730_gb300 import bddc
    return bddc


WL = {
    # blocks of 16 rows, bandwidth 16: L_{j,j-1} triangular
    "sub16": lambda: inputs.two_level_channels(nx=80, sub=16),
    # interiors of 16 x 16 and 8 x 8 nodes: bandwidth 17 and 9 in blocks of 16 and 8
    "sub17": lambda: inputs.two_level_channels(nx=68, sub=17),
    "sub9": lambda: inputs.two_level_channels(nx=72, sub=9),
    "cells": lambda: inputs.three_level_voronoi(nx=72, cells=4, group=2, levels=2),
    # 4 x 4 elements: more substructures than an SM's warps on a small mesh
    "sub4": lambda: inputs.two_level_channels(nx=100, sub=4),
    # edges of 71 nodes: the eigenproblems do not fit in shared memory
    "sub72": lambda: inputs.two_level_channels(nx=144, sub=72),
}
_cache = {}


def _oracle(name):
    if name not in _cache:
        wl = WL[name]()
        _cache[name] = (wl, obddc.build_workload(wl))
    return _cache[name]


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


# stream: the half-block ring kernel; lane: a lane per right-hand side
ROUTES = {"tuned": {}, "stream": {"BDDC_BATCH_STREAM": "1", "BDDC_TC": "0"},
          "lane": {"BDDC_DIR_LANE": "1", "BDDC_TC": "0"}}


@pytest.mark.parametrize("route", list(ROUTES))
@pytest.mark.parametrize("name", ["sub16", "sub17", "sub9", "cells", "sub4"])
def test_batch_widths_and_blocks(lib, monkeypatch, name, route):
    """Batches of 1 to 32 columns on each Dirichlet kernel: FP64 and FP32
    applies, and solves with the stencil's tile (up to 24 columns) and
    marching (from 25) forms."""
    for k, v in ROUTES[route].items():
        monkeypatch.setenv(k, v)
    wl, H = _oracle(name)
    R = inputs.normal_rhs(wl.n_dof, 61, 32)
    ref = [H.apply(r) for r in R]
    P = lib.Problem.from_workload(wl)
    try:
        for prec, tol in (("fp64", 1e-10), ("fp32", 1e-5)):
            P.set_precision(prec)
            for K in (3, 16, 17, 31, 32):
                Z = P.apply(torch.tensor(R[:K], device="cuda")).cpu().numpy()
                for j in range(K):
                    assert _rel(Z[j], ref[j]) <= tol, (prec, K, j)
        P.set_precision("fp64")
        for K in (2, 24, 25, 32):
            _, infos = P.solve(torch.tensor(R[:K], device="cuda"), rtol=1e-8)
            assert all(i["status"] == 0 and i["relres_true"] <= 1e-8 for i in infos), K
    finally:
        P.close()


@pytest.mark.parametrize("name", ["sub16", "sub17", "sub72", "cells"])
@pytest.mark.parametrize("generic", [False, True])
def test_single_column(lib, monkeypatch, name, generic):
    """One right-hand side: the warp kernels (generic: the block-per-
    substructure ones with their half-block ring), and the setup's edge
    eigenproblems in shared and in global memory."""
    if generic:
        monkeypatch.setenv("BDDC_GENERIC_DIR", "1")
    wl, H = _oracle(name)
    r = inputs.normal_rhs(wl.n_dof, 71)
    ref = H.apply(r)
    P = lib.Problem.from_workload(wl)
    try:
        for prec, tol in (("fp64", 1e-10), ("fp32", 1e-5)):
            P.set_precision(prec)
            assert _rel(P.apply(torch.tensor(r, device="cuda")).cpu().numpy(), ref) <= tol, prec
    finally:
        P.close()


def test_large_interiors_warp_kernel(lib):
    """169 elasticity substructures of 450 interior DOFs: FP32 and BF16 run the
    warp Dirichlet kernel that reads its records in rounds, FP64 the block
    kernel, which is the reference here."""
    wl = inputs.elasticity(nx=208, sub=16, constraints="corners+edges")
    r = torch.tensor(inputs.normal_rhs(wl.n_dof, 81), device="cuda")
    P = lib.Problem.from_workload(wl)
    try:
        ref = P.apply(r).cpu().numpy()
        for prec, tol in (("fp32", 1e-5), ("bf16", 1e-2)):
            P.set_precision(prec)
            assert _rel(P.apply(r).cpu().numpy(), ref) <= tol, prec
            _, (info,) = P.solve(torch.tensor(wl.rhs(), device="cuda"))
            assert info["status"] == 0 and info["relres_true"] <= 1e-8
    finally:
        P.close()


@pytest.mark.parametrize("bmin", [1, 33, 160, 200])
def test_top_factor_block_sizes(lib, monkeypatch, bmin):
    """Top-level blocks below and above what the factorisation kernel and the
    sixteen-lane rows of the sweeps take, without the dense inverse."""
    monkeypatch.setenv("BDDC_TOP_DENSE_MAX", "0")
    monkeypatch.setenv("BDDC_TOP_BMIN", str(bmin))
    wl, H = _oracle("sub4")
    R = inputs.normal_rhs(wl.n_dof, 91, 3)
    P = lib.Problem.from_workload(wl)
    try:
        for K in (1, 3):
            Z = P.apply(torch.tensor(R[:K], device="cuda")).cpu().numpy()
            for j in range(K):
                assert _rel(Z[j], H.apply(R[j])) <= 1e-10, (K, j)
    finally:
        P.close()
