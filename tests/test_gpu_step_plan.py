"""lbm_step_plan says which kernels lbm_step launches: the sizes at which the bitwise tests compare the
multi-step kernels with single steps do reach those kernels."""
import pytest

from tests import test_gpu_pairs as pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_7239_gb300 import build, lbm

    build.build()
    return lbm


def plan(lbm, nx, ny, bc_x=1, bc_y=1, n=10, het=0, thermal=0, **kw):
    if thermal:
        kw.update(thermal=1, tau_T=0.8, T0=11.0, T_wall=[21.0, 1.0, None, None])
    with lbm.Lattice(nx=nx, ny=ny, bc_x=bc_x, bc_y=bc_y, **kw) as lat:
        if het:
            import torch

            lat.set_medium(torch.full((ny, nx), 0.5, device="cuda"), None)
        return lat.step_plan(n)


@pytest.mark.parametrize("bc_x,bc_y", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_sizes_of_the_pair_tests_take_pairs(lbm, bc_x, bc_y):
    for nx, ny in pairs.SIZES:
        for prec, het, thermal in pairs.FLOW:
            assert plan(lbm, nx, ny, bc_x, bc_y, precision=prec, het=het, thermal=thermal)[0] == 2, (nx, ny, het, thermal)


def test_other_sizes_of_the_pair_tests(lbm):
    for nx, ny, bc_x, bc_y in [(4100, 3208, 0, 1), (3661, 3590, 1, 0), (3728, 3525, 1, 1)]:
        for prec in (1, 2):
            assert plan(lbm, nx, ny, bc_x, bc_y, precision=prec)[0] == 2
    for nx, ny, bc_y in [(1288, 1309, 1), (1289, 1308, 0), (1290, 1301, 1), (1303, 1290, 1)]:
        for het in (0, 1):
            assert plan(lbm, nx, ny, 2, bc_y, het=het)[0] == 2


@pytest.mark.parametrize("bc_x,bc_y", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_sizes_of_the_tile_tests_take_tiles(lbm, bc_x, bc_y):
    for nx, ny in [(16, 16), (61, 40), (64, 64), (65, 152), (120, 31), (121, 200), (513, 305)]:
        for prec, het, thermal in [(0, 0, 0), (0, 1, 0), (0, 0, 1), (1, 0, 0), (1, 1, 0), (1, 0, 1), (2, 0, 0)]:
            if bc_x == 0 and prec and nx % 4:  # (16-bit storage: whole groups of four cells)
                continue
            assert plan(lbm, nx, ny, bc_x, bc_y, precision=prec, het=het, thermal=thermal)[0] == 4, (nx, ny, prec, het, thermal)
    for nx, ny in [(16, 33), (65, 40), (122, 16), (211, 200)]:
        assert plan(lbm, nx, ny, 2, 1)[0] == 4


def test_kernels_of_a_call(lbm):
    assert plan(lbm, 64, 64, n=1) == (4, 1)
    assert plan(lbm, 64, 64, n=0) == (4, 0)
    assert plan(lbm, 64, 64, n=5) == (4, 2)  # four steps, the last one
    assert plan(lbm, 64, 64, n=8) == (4, 3)  # four, three, the last
    assert plan(lbm, 64, 64, n=7) == (4, 3)
    assert plan(lbm, 64, 64, n=6) == (4, 3)  # four, one, the last
    assert plan(lbm, 64, 64, n=129) == (4, 33)  # a graph of 32 launches, the last
    assert plan(lbm, 64, 64, n=256) == (4, 32 + 33)  # a graph, 31 launches of four, one of three, the last
    assert plan(lbm, 1500, 1500, n=5) == (2, 5)  # two pairs of two kernels, the last
    assert plan(lbm, 1500, 1500, n=4) == (2, 4)  # a pair, a step, the last
    assert plan(lbm, 1500, 1500, n=33) == (2, 33)  # a graph of sixteen pairs, the last
    assert plan(lbm, 130, 12700, n=3) == (2, 2)  # every strip has a side: one kernel a pair
    assert plan(lbm, 1000, 900, n=40) == (1, 40)  # between the two ranges
    assert plan(lbm, 2000, 2000, bc_x=3, bc_y=3, n=9) == (1, 9)
    assert plan(lbm, 2000, 2000, streaming=1, n=9) == (1, 9)
    assert plan(lbm, 64, 64, bc_x=3, bc_y=3, streaming=1, n=9) == (1, 18)  # the boundary nodes' kernel before each step
