"""The batched substructure correction at interfaces whose operator fits shared
memory only with small chunks: every column of a batched apply equals the single
right-hand-side one (FP64: 1e-10; FP32, the same rounded operators with FP32
sums: 1e-5), and a solve runs as one batch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_0911_5730_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0911_5730_gb300 import bddc
    return bddc


def _workload(nx, elem_to_sub, n_sub):
    return inputs.Workload("interfaces_%d" % nx, nx, inputs.constant_coefficient(nx),
                           np.asarray(elem_to_sub, dtype=np.int32), n_sub, 2, np.inf, "corners+edges")


def _strips(nx, w=16):
    """nx x nx elements in strips of w columns: interfaces of 2 (nx - 1) DOFs."""
    ei = np.arange(nx * nx) % nx
    return _workload(nx, ei // w, nx // w)


def _check(P, wl, prec, tol, K=4):
    P.set_precision(prec)
    R = torch.tensor(inputs.normal_rhs(wl.n_dof, 21, K), device="cuda")
    Z = P.apply(R)
    for k in range(K):
        z = P.apply(R[k])
        assert float(torch.linalg.norm(Z[k] - z) / torch.linalg.norm(z)) <= tol, (prec, k)
    _, infos = P.solve(R, rtol=1e-8)
    assert all(i["status"] == 0 and i["batch_width"] == K for i in infos), prec


def test_chunk_tuned_in_another_precision(lib, monkeypatch):
    """Chunks of 64 KB fit in FP32 (382 DOFs) and not in FP64."""
    monkeypatch.setenv("BDDC_NEU_CHUNK", str(64 * 1024))
    wl = _strips(192)
    P = lib.Problem.from_workload(wl, precision="fp32")
    try:
        _check(P, wl, "fp32", 1e-5)
        assert P.query(level=None)["tuned_neu_chunk"][0] == 64 * 1024
        _check(P, wl, "fp64", 1e-10)
    finally:
        P.close()


def _flanked(nx, per_side, w=16):
    """One strip of w columns with a grid of blocks on either side, three
    columns of per_side of them: the strip has an interface of 2 (nx - 1) DOFs
    with 2 per_side - 1 corners and edges a side."""
    ej, ei = np.divmod(np.arange(nx * nx), nx)
    x0 = (nx - w) // 2
    col = np.where(ei < x0, ei * 3 // x0, 3 + (ei - x0 - w) * 3 // (nx - x0 - w))
    blk = col * per_side + ej * per_side // nx
    return _workload(nx, np.where((ei >= x0) & (ei < x0 + w), 6 * per_side, blk), 6 * per_side + 1)


def test_small_chunk(lib):
    """502 DOFs and 14 coarse ones in FP64: two stages of 8 KB fit beside the
    record, two of 32 KB do not."""
    wl = _flanked(252, 4)
    P = lib.Problem.from_workload(wl)
    try:
        _check(P, wl, "fp64", 1e-10)
    finally:
        P.close()


@pytest.mark.parametrize("per_side,prec,tol", [(6, "fp64", 1e-10), (19, "fp32", 1e-5)])
def test_record_not_staged(lib, per_side, prec, tol):
    """502 DOFs with 22 (FP64) and 74 (FP32) coarse ones: the record leaves no
    room for the smallest chunks."""
    wl = _flanked(252, per_side)
    P = lib.Problem.from_workload(wl)
    try:
        _check(P, wl, prec, tol)
    finally:
        P.close()
