"""Steps taken in pairs (k_march) give bitwise the results of single steps (k_step), at widths and heights
around the strips and segments of the pair kernel and in every storage and medium it takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W = np.array([1 / 9] * 4 + [1 / 36] * 4, np.float32)[:, None, None]
FLOW = [(0, 0, 0), (0, 1, 0), (0, 0, 1)]  # (precision, per-cell medium, temperature) with states above 100 MB
SIZES = [(1288, 1309), (1449, 1137), (1211, 1360), (4100, 402), (130, 12700)]


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_7239_gb300 import build, lbm

    build.build()
    return lbm


def lattices(lbm, nx, ny, bc_x, bc_y, prec, het, thermal, n=2):
    import torch

    g = torch.Generator("cuda").manual_seed(nx + ny)
    kw = dict(thermal=1, tau_T=0.8, g_beta=1e-5, T0=11.0, T_wall=[21.0, 1.0, None, 5.0], dev_scale_log2=8) if thermal else {}
    out = []
    f = torch.tensor(1.5 * W, device="cuda") + 0.004 * torch.randn(8, ny, nx, generator=g, device="cuda")
    T = 2.2 + 0.2 * torch.randn(5, ny, nx, generator=g, device="cuda") if thermal else None
    eps = 0.3 + 0.5 * torch.rand(ny, nx, generator=g, device="cuda")
    K = torch.exp(2 + torch.rand(ny, nx, generator=g, device="cuda"))
    for _ in range(n):
        lat = lbm.Lattice(nx=nx, ny=ny, bc_x=bc_x, bc_y=bc_y, precision=prec, nu=0.05, phi=0.5, K=30.0, p_rest=0.5, ax=1e-5, ay=-2e-5,
                          u_wall=[(0, 0.02), (0, -0.01), (0.015, 0), (0.03, 0.005)], **kw)
        if het:
            lat.set_medium(eps, K)
        lat.set_populations(f, T)
        out.append(lat)
    return out


def compare(a, b, steps):
    import torch

    a.step(steps)
    for _ in range(steps):
        b.step(1)
    fa, fb = a.get_populations(), b.get_populations()
    for x, y in zip(fa if a.thermal else (fa,), fb if b.thermal else (fb,)):
        assert bool(torch.isfinite(y).all()) and torch.equal(x, y)
    assert a.residual() == b.residual() and a.step_count() == b.step_count()
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("bc_x,bc_y", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("prec,het,thermal", FLOW)
def test_pairs_equal_single_steps(lbm, nx, ny, bc_x, bc_y, prec, het, thermal):
    compare(*lattices(lbm, nx, ny, bc_x, bc_y, prec, het, thermal), steps=5)


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("nx,ny,bc_x,bc_y", [(4100, 3208, 0, 1), (3661, 3590, 1, 0), (3728, 3525, 1, 1)])
def test_pairs_equal_single_steps_16bit(lbm, prec, nx, ny, bc_x, bc_y):
    compare(*lattices(lbm, nx, ny, bc_x, bc_y, prec, 0, 0), steps=4)


def test_graph_of_pairs(lbm):
    """Runs of more than 32 steps (graphs of pairs), from either buffer."""
    a, b = lattices(lbm, 1300, 1301, 1, 1, 0, 0, 0)
    a.step(3)
    for _ in range(3):
        b.step(1)
    compare(a, b, steps=75)
