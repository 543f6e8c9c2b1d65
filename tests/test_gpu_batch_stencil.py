"""The batched stencil on both sides of the width from which it marches, with
every tile: FP32 solves whose true relative residual meets the tolerance."""
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


@pytest.mark.parametrize("variant,tile", list(enumerate([[16, 8], [32, 4], [32, 8], [8, 16]])))
def test_tiles_and_march(lib, monkeypatch, variant, tile):
    monkeypatch.setenv("BDDC_TILE_VARIANT", str(variant))
    wl = inputs.two_level_channels(nx=80, sub=16)
    B = torch.tensor(inputs.normal_rhs(wl.n_dof, 61, 32), device="cuda")
    P = lib.Problem.from_workload(wl, precision="fp32")
    try:
        for K in (2, 23, 24, 25, 32):
            _, infos = P.solve(B[:K].contiguous(), rtol=1e-8)
            assert all(i["status"] == 0 and i["relres_true"] <= 1e-8 for i in infos), K
        assert P.query(level=None)["tuned_tile"][:2] == tile
    finally:
        P.close()
