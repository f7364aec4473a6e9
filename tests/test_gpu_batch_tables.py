"""The work-item tables of a batch are replaced only after the steps in flight, which read them."""
import pytest

from paper_1311_7239_gb300 import workloads

pytestmark = pytest.mark.gpu


def test_tables_are_not_replaced_under_steps_in_flight():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_7239_gb300 import build, lbm

    build.build()
    cfgs, media = workloads.ensemble(lbm, n=9, seed=6, lo=64, hi=300)
    with workloads.build(lbm, cfgs, media) as a, workloads.build(lbm, cfgs, media) as b:
        for nt, tiling, items in [(64, lbm.TILING_ROWS, 1), (256, lbm.TILING_FLAT, 1), (128, lbm.TILING_ROWS, 2), (64, lbm.TILING_FLAT, 4)]:
            a.set_tiling(tiling)
            a.set_items_per_cta(items)
            a.set_launch(nt, 0)
            a.step(160)  # (five graphs, not waited for)
        b.step_each(640)
        a.sync()
        for d in range(len(cfgs)):
            assert torch.equal(a.get_populations(d), b.get_populations(d)), d
