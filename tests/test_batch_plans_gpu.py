"""Batch plans beside other plans of other sizes."""
import numpy as np
import pytest

import synth
from test_batched_gpu import _dev_scene, _run_single

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ex():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_29663_gb300 import build
    build.build()
    import paper_2605_29663_gb300 as ex
    return ex


def _scenes(sizes, shared, seed):
    g = synth.rng(seed)
    out = []
    for i, (K, T, N) in enumerate(sizes):
        s = synth.random_scene(g, [synth.DIFF, synth.OMNI][i % 2], 10, N, K, T, n_obst=20)
        if shared:
            s["kind"], s["fp"] = synth.POLYGON, synth.l_footprint()
        out.append(s)
    return out


def _check(ex, scenes, dev, b, dmin):
    import torch
    torch.cuda.synchronize()
    assert b.get_error() == 0
    ctx = ex.Context()
    for i, (s, d, o) in enumerate(zip(scenes, dev, b.outputs)):
        want = _run_single(ex, ctx, s, dmin=dmin)
        for k in ("costs", "weights", "U_upd", "u_star"):
            np.testing.assert_array_equal(o[k].cpu().numpy(), want[k], err_msg=f"scene {i} {k}")
        np.testing.assert_array_equal(d["U"].cpu().numpy(), want["U"], err_msg=f"scene {i} U")


@pytest.mark.parametrize("tune", [False, True])
@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("dmin", [False, True])
def test_an_older_plan_steps_after_a_newer_smaller_one(ex, dmin, shared, tune):
    """The largest shared memory first (long horizon and many samples; clouds
    that fill the stage), then a plan that needs little, tuned or not."""
    old = _scenes([(2500, 100, 4200), (700, 128, 2000)] if not dmin else [(200, 30, 5000), (100, 60, 4100)], shared, 5)
    new = _scenes([(40, 9, 60), (64, 10, 50)], shared, 6)
    dev = [_dev_scene(ex, s) for s in old]
    a = ex.Batch(dev, dmin=dmin)
    small = [_dev_scene(ex, s) for s in new]
    for other in (dmin, not dmin):
        b = ex.Batch(small, dmin=other)
        if tune:
            b.autotune(iters=1)
        b.step()
    a.step()
    _check(ex, old, dev, a, dmin)
