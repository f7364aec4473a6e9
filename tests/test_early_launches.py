"""Kernels that are launched while the kernel before them still runs read what that one writes only after
they have waited for it: by ordinary loads, never as memory that is constant while they live."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1311_7239_gb300", "csrc")
# parameters that only the host writes, with no kernel of the library in flight
TABLES = {"R", "Pd", "item_start", "item_lattice", "items"}


def _sources():
    return {os.path.basename(p): open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}


def test_wall_velocities_are_not_read_through_the_read_only_path():
    for name, text in _sources().items():
        assert not re.search(r"__ld\w+\([^;]*\buw\b", text), name


def test_early_kernels_have_no_restrict_parameter_but_tables():
    found = 0
    for name, text in _sources().items():
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(([^{;]*)\)\s*\{", text):
            body = text[m.end(): text.index("\n}", m.end())]
            if "wait_prerequisites()" not in body:
                continue
            found += 1
            for p in m.group(2).split(","):
                if "__restrict__" in p:
                    assert re.search(r"(\w+)\s*$", p).group(1) in TABLES, (name, m.group(1), p)
    assert found >= 7


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("bc", [1, 3])
@pytest.mark.parametrize("nx,ny,steps", [(1024, 1024, 1), (1283, 1024, 1), (100, 80, 5), (96, 1024, 5)])
def test_new_walls_reach_the_next_step(nx, ny, steps, bc, prec):
    """Walls from page-locked memory, a step, a probe beside the lid, over and over without a wait, give the
    bits of a context that waits after every call."""
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_7239_gb300 import build, lbm

    build.build()
    n = 24
    walls = torch.zeros(n, 4, 2)
    walls[:, 3, 0] = 0.1 * (-1.0) ** torch.arange(n)  # the lid turns round before every step
    walls[:, 2, 0] = 0.05 * (-1.0) ** (torch.arange(n) // 2)
    walls[:, 0, 1] = 0.03 * torch.cos(torch.arange(n).float())
    walls, out = walls.pin_memory(), []
    for wait in (True, False):
        probe = torch.zeros(n, 4).pin_memory()
        with lbm.Lattice(nx=nx, ny=ny, bc_x=bc, bc_y=bc, precision=prec, nu=0.1, phi=0.5, K=100.0, p_rest=0.5) as lat:
            lat.init_equilibrium(1.0, 0.0, 0.0)
            for k in range(n):
                lat.set_walls(walls[k])
                if wait:
                    lat.sync()
                lat.step(steps)
                if wait:
                    lat.sync()
                lat.probe_async(nx // 2, ny - 2, probe[k])
                if wait:
                    lat.sync()
            f = lat.get_populations()
            lat.sync()
        out.append((probe, f))
    assert bool((out[0][0][1:, 1] != out[0][0][:-1, 1]).all())
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
