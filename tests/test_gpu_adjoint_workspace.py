"""The workspace that lbm_adjoint keeps serves calls of a somewhat smaller T, as in a run whose T changes
from call to call, and is made anew where it would be more than twice what the call needs."""
import pytest

pytestmark = pytest.mark.gpu


def test_workspace_serves_smaller_calls():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_7239_gb300 import build, lbm

    build.build()
    nx, ny = 96, 64

    def call(lat, T):
        lat.init_equilibrium(1.0, 0.0, 0.0)
        out = lat.adjoint(T, "flux")
        return out, lat.memory_bytes()

    kw = dict(nx=nx, ny=ny, bc_x=lbm.PRESSURE, bc_y=lbm.WALL, nu=0.1, phi=0.5, K=50.0, p_rest=0.5, p_in=1.002, p_out=0.998)
    for streaming in (lbm.STREAM_AB, lbm.STREAM_INPLACE):
        with lbm.Lattice(streaming=streaming, **kw) as lat, lbm.Lattice(streaming=streaming, **kw) as fresh:
            (_, held) = call(lat, 100)
            for T in (81, 100, 64):
                (L, gk, ge), now = call(lat, T)
                assert now == held, T
                fresh.release_workspace()
                (Lf, gkf, gef), _ = call(fresh, T)
                assert L == Lf and torch.equal(gk, gkf) and torch.equal(ge, gef), T
            assert call(lat, 4)[1] < held
            assert call(lat, 100)[1] == held
