"""Launch shapes and steps per launch of batches that can take their steps in pairs: a chosen shape is the
one that runs, the tuner times pairs beside the shapes, and neither changes a bit."""
import json

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_7239_gb300 import build, lbm

    build.build()
    return lbm


SHAPES = [(640, 701, 1), (503, 512, 0), (801, 600, 1), (700, 640, 0), (512, 512, 1), (655, 599, 1)]  # above 100 MB


def batch(lbm, shapes=SHAPES, **kw):
    b = lbm.Batch([lbm.default_config(nx=nx, ny=ny, bc_x=bx, bc_y=1, nu=0.06, phi=0.45, K=20.0, p_rest=0.45, ax=0.0 if bx else 1e-5,
                                      u_wall=[(0, 0), (0, 0), (0, 0), (0.02, 0)], **kw) for nx, ny, bx in shapes])
    b.init_equilibrium(-1, 1.0, 0.0, 0.0)
    return b


def state(b):
    b.sync()
    return [b.get_populations(d) for d in range(len(b))]


def test_a_chosen_launch_shape_runs(lbm):
    import torch

    with batch(lbm) as a, batch(lbm) as b:
        assert a.get_steps_per_launch() == 2
        for choose in (lambda: a.set_launch(128, 4), lambda: a.set_items_per_cta(2), lambda: a.set_tiling(lbm.TILING_ROWS)):
            a.set_steps_per_launch(2)
            a.step(37)
            choose()
            assert a.get_steps_per_launch() == 1
            a.step(35)
        b.step_each(3 * (37 + 35))
        assert all(torch.equal(x, y) for x, y in zip(state(a), state(b)))
        with pytest.raises(lbm.LbmError):
            a.set_steps_per_launch(3)


def test_tuner_times_pairs(lbm):
    import torch

    with batch(lbm) as a, batch(lbm) as b:
        nt, k, ms = a.tune(steps=4)
        chosen = a.get_steps_per_launch()
        assert chosen in (1, 2) and ms > 0 and a.get_launch() == (nt, k)
        a.step(33)
        b.step_each(33)
        assert all(torch.equal(x, y) for x, y in zip(state(a), state(b)))


def test_batches_without_pairs(lbm):
    for b in (batch(lbm, [(100, 90, 1), (64, 300, 0)]), batch(lbm, precision=lbm.FP16_DEV), batch(lbm, streaming=lbm.STREAM_INPLACE)):
        with b:
            assert b.get_steps_per_launch() == 1
            b.set_steps_per_launch(1)
            with pytest.raises(lbm.LbmError):
                b.set_steps_per_launch(2)


def test_tuning_cache_keeps_steps_per_launch(lbm, tmp_path):
    path = str(tmp_path / "tune.json")
    with batch(lbm) as a:
        a.tune_cached(path, steps=4)
        chosen = a.get_steps_per_launch()
    with batch(lbm) as a:
        assert a.tune_cached(path, steps=4)[3] and a.get_steps_per_launch() == chosen
    cache = json.load(open(path))
    for v in cache.values():
        assert v.pop("steps_per_launch") == chosen
    json.dump(cache, open(path, "w"))  # an entry without it: the batch keeps its own choice
    with batch(lbm) as a:
        assert a.tune_cached(path, steps=4)[3] and a.get_steps_per_launch() == 2
