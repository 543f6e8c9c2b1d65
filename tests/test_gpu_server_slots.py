"""A server slot whose last right-hand side was not a number, or infinite, serves
the next one as if it were new."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_0911_5730_gb300 import inputs  # noqa: E402


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_slot_after_nan(precision, value):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0911_5730_gb300 import bddc
    wl = inputs.two_level_channels(nx=80, sub=16)
    P = bddc.Problem.from_workload(wl, precision=precision)
    srv = bddc.Server()
    try:
        # as many columns as the engines of one problem have slots, twice over
        bad = np.full((192, wl.n_dof), value)
        srv.wait(srv.submit(P, bad, maxit=3))
        _, infos, _ = srv.wait(srv.submit(P, inputs.normal_rhs(wl.n_dof, 31, 192)))
        assert all(i["status"] == 0 and i["relres_true"] <= 1e-8 for i in infos)
    finally:
        srv.close()
        P.close()
