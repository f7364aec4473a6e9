"""Steps taken in pairs (k_march) or four at a time in shared memory (k_tile) give bitwise the results of
single steps (k_step), at widths and heights around the strips, segments and tiles of those kernels and in
every storage, medium and side that they take."""
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


def lattices(lbm, nx, ny, bc_x, bc_y, prec, het, thermal, n=2, amp=0.004):
    import torch

    g = torch.Generator("cuda").manual_seed(nx + ny)
    kw = dict(thermal=1, tau_T=0.8, g_beta=1e-5, T0=11.0, T_wall=[21.0, 1.0, None, 5.0], dev_scale_log2=8) if thermal else {}
    out = []
    f = torch.tensor(1.5 * W, device="cuda") + amp * torch.randn(8, ny, nx, generator=g, device="cuda")
    T = 2.2 + 0.2 * torch.randn(5, ny, nx, generator=g, device="cuda") if thermal else None
    eps = 0.3 + (0.1 if bc_x == 2 else 0.5) * torch.rand(ny, nx, generator=g, device="cuda")
    K = torch.exp(2 + torch.rand(ny, nx, generator=g, device="cuda"))
    for _ in range(n):
        lat = lbm.Lattice(nx=nx, ny=ny, bc_x=bc_x, bc_y=bc_y, precision=prec, nu=0.05, phi=0.5, K=30.0, p_rest=0.5, ax=1e-5, ay=-2e-5, p_in=1.01, p_out=0.99,
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


@pytest.mark.parametrize("het", [0, 1])
@pytest.mark.parametrize("nx,ny,bc_y", [(1288, 1309, 1), (1289, 1308, 0), (1290, 1301, 1), (1303, 1290, 1)])
def test_pairs_with_pressure_columns(lbm, nx, ny, bc_y, het):
    compare(*lattices(lbm, nx, ny, 2, bc_y, 0, het, 0, amp=0.001), steps=5)


# (several steps per launch in shared memory: one, two and more tiles wide, one or more rows per tile,
# the last tile one column or row wide)
@pytest.mark.parametrize("nx,ny", [(16, 16), (61, 40), (64, 64), (65, 152), (120, 31), (121, 200), (513, 305)])
@pytest.mark.parametrize("prec,het,thermal", [(0, 0, 0), (0, 1, 0), (0, 0, 1), (1, 0, 0), (1, 1, 0), (1, 0, 1), (2, 0, 0)])
@pytest.mark.parametrize("bc_x,bc_y", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_tiles_equal_single_steps(lbm, nx, ny, prec, het, thermal, bc_x, bc_y):
    compare(*lattices(lbm, nx, ny, bc_x, bc_y, prec, het, thermal), steps=12)


@pytest.mark.parametrize("het", [0, 1])
@pytest.mark.parametrize("nx,ny", [(16, 33), (65, 40), (122, 16), (211, 200)])
def test_tiles_with_pressure_columns(lbm, nx, ny, het):
    compare(*lattices(lbm, nx, ny, 2, 1, 0, het, 0, amp=0.0005), steps=7)


def test_tile_graphs(lbm):
    compare(*lattices(lbm, 150, 70, 1, 1, 0, 1, 0), steps=400)


def test_batched_pairs_equal_single_lattices(lbm):
    """A batch above 100 MB takes its steps in pairs; each lattice ends on the bits of its own context."""
    import torch

    shapes = [(1024, 700, 1), (61, 900, 0), (129, 64, 1), (64, 130, 1), (997, 803, 0), (16, 16, 0), (301, 257, 1)]
    g = torch.Generator("cuda").manual_seed(4)
    cfgs, media = [], []
    for nx, ny, wall in shapes:
        cfgs.append(lbm.default_config(nx=nx, ny=ny, bc_x=wall, bc_y=1, nu=0.06, phi=0.45, K=20.0, p_rest=0.45, ax=0.0 if wall else 1e-5,
                                       u_wall=[(0, 0), (0, 0), (0, 0), (0.02, 0)]))
        media.append((0.3 + 0.4 * torch.rand(ny, nx, generator=g, device="cuda"), torch.exp(2 + torch.rand(ny, nx, generator=g, device="cuda"))))
    with lbm.Batch(cfgs) as b:
        for d, (eps, K) in enumerate(media):
            b.set_medium(d, eps, K)
            b.init_equilibrium(d, 0.45, 0.0, 0.0, phi_p_uniform=True)
        b.step(32 + 7)  # a graph of pairs, three pairs, a single step
        b.step(2)
        b.sync()
        assert b.info()["steps"] == 41
        for d, (eps, K) in enumerate(media):
            with lbm.Lattice(lbm.Config.from_buffer_copy(cfgs[d])) as lat:
                lat.set_medium(eps, K)
                lat.init_equilibrium(0.45, 0.0, 0.0, phi_p_uniform=True)
                for _ in range(41):
                    lat.step(1)
                assert torch.equal(b.get_populations(d), lat.get_populations()), d
