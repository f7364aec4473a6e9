"""The kernels that take several steps per launch check their index invariants in the debug build as the
others do (a violation sets an error bit, which the next synchronising call reports, and the access is
skipped): small lattices of every form that k_tile takes, lattices above the size of L2 (k_march,
k_march_side), and a batch of them (k_march_batch)."""
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1311_7239_gb300", "csrc")

SCRIPT = r'''
import itertools
import torch
from paper_1311_7239_gb300 import lbm, workloads

def run(nx, ny, bx, by, prec, het, thermal, steps, sv=False):
    kw = dict(thermal=1, tau_T=0.8, g_beta=1e-5, T0=11.0, T_wall=[21.0, 1.0, None, 5.0], dev_scale_log2=8) if thermal else {}
    with lbm.Lattice(nx=nx, ny=ny, bc_x=bx, bc_y=by, precision=prec, nu=0.05, phi=0.5, K=30.0, p_rest=0.5, ax=1e-5, p_in=1.001, p_out=0.999,
                     u_wall=[(0, 0.01), (0, 0), (0, 0), (0.05, 0)], **kw) as lat:
        if het:
            lat.set_medium(torch.full((ny, nx), 0.5, device="cuda"), torch.full((ny, nx), 20.0, device="cuda"))
        if sv:
            lat.set_viscosity_ratio(torch.full((ny, nx), 1.5, device="cuda"))
        lat.init_equilibrium(0.5, 0.0, 0.0, phi_p_uniform=True)
        for n in steps:
            lat.step(n)
        lat.sync()

FORMS = [(0, 0, 0), (0, 1, 0), (0, 0, 1), (1, 0, 0), (1, 1, 0), (1, 0, 1), (2, 0, 0), (2, 1, 0), (2, 0, 1)]  # (precision, per-cell medium, temperature)
SIDES = [(0, 0), (0, 1), (1, 0), (1, 1)]
runs = 0
for nx, ny in [(16, 16), (61, 40), (64, 64), (65, 152), (120, 31), (121, 200), (316, 40), (513, 305)]:
    for (prec, het, thermal), (bx, by) in itertools.product(FORMS, SIDES):
        run(nx, ny, bx, by, prec, het, thermal, (9, 2, 3, 4))
        runs += 1
    for het, by in itertools.product((0, 1), (0, 1)):
        run(nx, ny, 2, by, 0, het, 0, (9, 2))
    run(nx, ny, 1, 1, 0, 1, 0, (7,), sv=True)
for nx, ny in [(1288, 1309), (1449, 1137), (4100, 402), (130, 12700)]:
    for (het, thermal), (bx, by) in itertools.product([(0, 0), (1, 0), (0, 1)], SIDES):
        run(nx, ny, bx, by, 0, het, thermal, (5,))
        runs += 1
    for het, by in itertools.product((0, 1), (0, 1)):
        run(nx, ny, 2, by, 0, het, 0, (5,))
    run(nx, ny, 1, 1, 0, 1, 0, (5,), sv=True)
for prec, (nx, ny, bx, by) in itertools.product((1, 2), [(4100, 3208, 0, 1), (3661, 3590, 1, 0), (3728, 3525, 1, 1), (4100, 3208, 0, 0)]):
    run(nx, ny, bx, by, prec, 0, 0, (5,))
    runs += 1
cfgs = [lbm.default_config(nx=nx, ny=ny, bc_x=bx, bc_y=by, nu=0.06, phi=0.45, K=20.0, p_rest=0.45, p_in=1.001, p_out=0.999)
        for nx, ny, bx, by in [(1024, 700, 1, 1), (61, 900, 0, 0), (129, 64, 1, 1), (64, 130, 1, 0), (997, 803, 2, 1), (16, 16, 0, 1), (301, 257, 0, 1)]]
with lbm.Batch(cfgs) as b:
    b.step(32 + 5)
    b.sync()
print("runs", runs)
'''


def test_every_step_kernel_checks_its_indices():
    for name in ("step.cu", "inplace.cu", "adjoint.cu", "march.cu", "tile.cu", "rows.cuh"):
        assert re.search(r"\bdbg_check\(", open(os.path.join(CSRC, name)).read()), name


@pytest.mark.gpu
def test_debug_build_of_the_multi_step_kernels_reports_no_violation():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_7239_gb300 import build

    env = dict(os.environ, LBM_LIBRARY=build.build(debug=True), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", SCRIPT], env=env, capture_output=True, text=True, timeout=900, cwd=ROOT)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "runs" in r.stdout
