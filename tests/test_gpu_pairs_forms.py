"""Forms of the multi-step kernels beside those of test_gpu_pairs.py: bitwise the results of single steps
with a per-cell viscosity ratio, with pressure columns in a batch, and between pressure columns and
periodic rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W = np.array([1 / 9] * 4 + [1 / 36] * 4, np.float32)[:, None, None]


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_7239_gb300 import build, lbm

    build.build()
    return lbm


def twins(lbm, nx, ny, bc_x, bc_y, het=0, ratio=0, prec=0, amp=0.002):
    """Two lattices in the same random state."""
    import torch

    g = torch.Generator("cuda").manual_seed(3 * nx + ny)
    f = torch.tensor(1.5 * W, device="cuda") + amp * torch.randn(8, ny, nx, generator=g, device="cuda")
    eps = 0.3 + 0.1 * torch.rand(ny, nx, generator=g, device="cuda")
    K = torch.exp(2 + torch.rand(ny, nx, generator=g, device="cuda"))
    J = 1.0 + 2.0 * torch.rand(ny, nx, generator=g, device="cuda")
    out = []
    for _ in range(2):
        lat = lbm.Lattice(nx=nx, ny=ny, bc_x=bc_x, bc_y=bc_y, precision=prec, nu=0.05, phi=0.5, K=30.0, p_rest=0.5, ax=1e-5, ay=-2e-5,
                          p_in=1.01, p_out=0.99, u_wall=[(0, 0.02), (0, -0.01), (0.015, 0), (0.03, 0.005)])
        if het:
            lat.set_medium(eps, K)
        if ratio:
            lat.set_viscosity_ratio(J)
        lat.set_populations(f)
        out.append(lat)
    return out


def compare(a, b, steps):
    import torch

    with a, b:
        a.step(steps)
        for _ in range(steps):
            b.step(1)
        fa, fb = a.get_populations(), b.get_populations()
        assert bool(torch.isfinite(fa).all()) and torch.equal(fa, fb)
        assert a.residual() == b.residual()


@pytest.mark.parametrize("nx,ny", [(1288, 1309), (1449, 1137), (61, 40), (121, 200)])
@pytest.mark.parametrize("bc_x,bc_y", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_viscosity_ratio(lbm, nx, ny, bc_x, bc_y):
    compare(*twins(lbm, nx, ny, bc_x, bc_y, het=1, ratio=1), steps=6)


@pytest.mark.parametrize("het", [0, 1])
@pytest.mark.parametrize("nx,ny", [(16, 33), (65, 40), (122, 16), (211, 200), (1289, 1308)])
def test_pressure_columns_with_periodic_rows(lbm, nx, ny, het):
    compare(*twins(lbm, nx, ny, 2, 0, het=het, amp=0.0005), steps=7)


def test_pressure_columns_in_a_paired_batch(lbm):
    import torch

    shapes = [(801, 700, 2, 1), (603, 902, 2, 0), (129, 640, 1, 1), (640, 331, 2, 1), (997, 803, 0, 1), (700, 500, 2, 1)]
    g = torch.Generator("cuda").manual_seed(5)
    cfgs, media = [], []
    for nx, ny, bx, by in shapes:
        cfgs.append(lbm.default_config(nx=nx, ny=ny, bc_x=bx, bc_y=by, nu=0.06, phi=0.45, K=20.0, p_rest=0.45, p_in=1.005, p_out=0.995,
                                       u_wall=[(0, 0), (0, 0), (0, 0), (0.02, 0)]))
        media.append((0.4 + 0.05 * torch.rand(ny, nx, generator=g, device="cuda"), torch.exp(2 + torch.rand(ny, nx, generator=g, device="cuda"))))
    steps = 32 + 5
    with lbm.Batch(cfgs) as b:
        for d, (eps, K) in enumerate(media):
            b.set_medium(d, eps, K)
            b.init_equilibrium(d, 0.45, 0.0, 0.0, phi_p_uniform=True)
        b.step(steps)
        b.sync()
        for d, (eps, K) in enumerate(media):
            with lbm.Lattice(lbm.Config.from_buffer_copy(cfgs[d])) as lat:
                lat.set_medium(eps, K)
                lat.init_equilibrium(0.45, 0.0, 0.0, phi_p_uniform=True)
                for _ in range(steps):
                    lat.step(1)
                assert torch.equal(b.get_populations(d), lat.get_populations()), d


@pytest.mark.parametrize("T", [7, 12])
def test_adjoint_of_a_large_in_place_context(lbm, T):
    """The forward sweep in pairs (above 100 MB), with T off and on the checkpoint interval: an in-place
    context gives the loss, the gradients and the final state of an A-B one, which are those of steps taken
    one at a time."""
    import torch

    nx, ny = 1449, 1137
    g = torch.Generator("cuda").manual_seed(8)
    eps = 0.4 + 0.02 * torch.rand(ny, nx, generator=g, device="cuda")
    K = torch.exp(3 + 0.5 * torch.rand(ny, nx, generator=g, device="cuda"))
    got = []
    for streaming in (lbm.STREAM_AB, lbm.STREAM_INPLACE):
        with lbm.Lattice(nx=nx, ny=ny, bc_x=lbm.PRESSURE, bc_y=lbm.WALL, nu=0.1, phi=0.4, K=30.0, p_rest=0.4, p_in=1.002, p_out=0.998,
                         streaming=streaming) as lat:
            lat.set_medium(eps, K)
            lat.init_equilibrium(0.4, 0.0, 0.0, phi_p_uniform=True)
            L, gk, ge = lat.adjoint(T, "flux")
            got.append((L, gk, ge, lat.get_populations(), lat.residual()))
    a, b = got
    assert a[0] == b[0] and all(torch.equal(x, y) for x, y in zip(a[1:4], b[1:4]))
    with lbm.Lattice(nx=nx, ny=ny, bc_x=lbm.PRESSURE, bc_y=lbm.WALL, nu=0.1, phi=0.4, K=30.0, p_rest=0.4, p_in=1.002, p_out=0.998) as lat:
        lat.set_medium(eps, K)
        lat.init_equilibrium(0.4, 0.0, 0.0, phi_p_uniform=True)
        for _ in range(T):
            lat.step(1)
        assert torch.equal(lat.get_populations(), a[3]) and lat.residual() == a[4]
