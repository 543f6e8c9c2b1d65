"""Batches on a level whose substructures have blocks of very different sizes:
four 40 x 40 cells with a small patch where they meet, so that no uniform block
size exists and every substructure streams with its own smallest one (1 to 5
rows in the patch, 39 and 40 beside it).

FP64 and FP32 applies are compared with the CPU oracle at the parity
tolerances (1e-10, 1e-5).  A BF16 apply is compared with the single
right-hand-side apply of the same rounded operators: both accumulate in FP32,
so they may differ as an FP32 apply may, by 1e-5.
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


def _patched(p, nx=80):
    e2s, _ = inputs.grid_decomposition(nx, nx // 2)
    e = e2s.reshape(nx, nx).copy()
    a = nx // 2 - p // 2
    e[a:a + p, a:a + p] = 4
    return inputs.Workload("patched_%d" % p, nx, inputs.channel_coefficient(nx, 2001),
                           e.reshape(-1).astype(np.int32), 5, 2, 10.0, "adaptive")


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("p", [6, 3, 2])      # interiors of 5 x 5, 2 x 2 and 1 x 1 nodes
def test_small_blocks_beside_large_ones(lib, p):
    wl = _patched(p)
    assert lib.inspect(wl.nx, wl.elem_to_sub, wl.n_sub1)["block_size"] == 0
    H = obddc.build_workload(wl)
    R = inputs.normal_rhs(wl.n_dof, 51, 32)
    ref = [H.apply(r) for r in R]
    P = lib.Problem.from_workload(wl)
    try:
        for prec, tol in (("fp64", 1e-10), ("fp32", 1e-5), ("bf16", 1e-5)):
            P.set_precision(prec)
            if prec == "bf16":
                ref = [P.apply(torch.tensor(r, device="cuda")).cpu().numpy() for r in R]
            for K in (2, 5, 32):
                Z = P.apply(torch.tensor(R[:K], device="cuda")).cpu().numpy()
                for j in range(K):
                    assert _rel(Z[j], ref[j]) <= tol, (prec, K, j)
    finally:
        P.close()
