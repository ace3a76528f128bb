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


def _mixed_batch(ex, scenes, dev, dmin):
    """A batch whose scene i has a d_min output when dmin[i]."""
    import ctypes
    arr, outputs, keep = ex._scene_array(dev, True, True, True, True, False)
    for i, want in enumerate(dmin):
        if not want:
            arr[i].dmin = None
            outputs[i].pop("dmin")
    h = ctypes.c_void_p()
    ex._check(ex.load().exact_batch_create(len(dev), ctypes.cast(arr, ctypes.c_void_p), ctypes.byref(h)), "create")
    b = ex.Batch.__new__(ex.Batch)
    b._h, b.n, b.outputs, b._keep, b.class_key = h, len(dev), outputs, keep, ""
    return b


def _check(ex, scenes, dev, b, dmin):
    import torch
    torch.cuda.synchronize()
    assert b.get_error() == 0
    ctx = ex.Context()
    dmin = dmin if isinstance(dmin, list) else [dmin] * len(scenes)
    for i, (s, d, o) in enumerate(zip(scenes, dev, b.outputs)):
        want = _run_single(ex, ctx, s, dmin=dmin[i])
        for k in ("costs", "weights", "U_upd", "u_star") + (("dmin",) if "dmin" in o else ()):
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


@pytest.mark.parametrize("shared", [False, True])
def test_autotune_times_what_a_step_runs(ex, shared):
    """A d_min output switches every pruning off: the tuner must time that, not
    the pruned cycle.  Points a metre and more beyond d_safe, so that pruned the
    sample phase would do next to nothing: its times are those of the step, of
    which it is all but a few us (a third is left for noise).  The scenes' d_min
    is not written, and block sizes are all that varies."""
    import torch
    scenes = _scenes([(1500, 20, 6000)] * 6, shared, 8)
    g = synth.rng(2)
    for s in scenes:
        a = g.uniform(-np.pi, np.pi, 6000)
        s["cloud"], s["mask"] = (np.stack([np.cos(a), np.sin(a)], 1) * g.uniform(8, 12, (6000, 1))).astype(np.float32), None
        s["q0"], s["U"] = np.zeros(3, np.float32), s["U"] * 0
    b = ex.Batch([_dev_scene(ex, s) for s in scenes], dmin=True)
    for o in b.outputs:
        o["dmin"].fill_(-7.0)
    report = b.autotune(iters=3)
    assert all(bool((o["dmin"] == -7.0).all()) for o in b.outputs)
    assert {c["threads"] for c in report["candidates"]} == {128, 256, 512}
    assert len({c["pairs_per_lane"] for c in report["candidates"]}) == 1
    b.step()
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    e[0].record()
    for _ in range(5):
        b.step()
    e[1].record()
    torch.cuda.synchronize()
    step = e[0].elapsed_time(e[1]) / 5
    assert report["best"]["ms"] > step / 3, (report["best"], step)
    assert all(bool((o["dmin"] > 0).all()) for o in b.outputs)


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("sizes,dmin", [
    ([(100, 20, 300), (64, 12, 1023), (200, 33, 900)], [0, 0, 0]),                  # few samples: items
    ([(1500, 32, 100), (700, 20, 1), (300, 60, 599)], [0, 0, 0]),                   # many: grids
    ([(1500, 33, 100), (700, 60, 400), (300, 20, 600)], [0, 0, 0]),                 # many, most of them not paying: items
    ([(100, 20, 300), (64, 12, 1024), (200, 33, 0)], [0, 0, 0]),                    # beside a grid
    ([(100, 20, 300), (64, 12, 700), (3000, 20, 800)], [1, 0, 0]),                  # beside d_min scenes: items
    ([(100, 20, 300), (64, 12, 3000), (3000, 20, 800), (50, 9, 5000)], [1, 0, 0, 1]),   # beside both, many: grids
    ([(100, 20, 300), (64, 12, 3000), (30, 20, 800), (50, 9, 5000)], [1, 0, 0, 1])])    # beside both, few: items
def test_scenes_of_every_route_in_one_batch(ex, sizes, dmin, shared):
    """Small scenes as items or on grids, alone, beside scenes that walk one and
    beside scenes with a d_min output: each gives its single-scene bits, twice in
    a row, whatever the block size."""
    import torch
    scenes = _scenes(sizes, shared, len(sizes) + sum(dmin))
    for tiles in (None, (64, 8), (512, 1)):
        dev = [_dev_scene(ex, s) for s in scenes]
        b = _mixed_batch(ex, scenes, dev, dmin)
        if tiles:
            b.set_tiles(*tiles)
        b.step()
        _check(ex, scenes, dev, b, [bool(d) for d in dmin])
        for s, d in zip(scenes, dev):
            d["U"].copy_(torch.from_numpy(s["U"]))
        b.step()
        _check(ex, scenes, dev, b, [bool(d) for d in dmin])


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("T", [33, 64, 65])
def test_smallest_block_with_two_samples_per_item(ex, T, shared):
    """64 threads, with enough samples for two per item (and, at T = 65, not):
    the warps that roll the two out leave none to stage the points."""
    scenes = _scenes([(700, T, 300), (101, 20, 1200)], shared, T)
    dev = [_dev_scene(ex, s) for s in scenes]
    b = ex.Batch(dev, dmin=True)
    b.set_tiles(64, 1)
    b.step()
    _check(ex, scenes, dev, b, True)


def test_batch_with_a_safety_distance_beyond_the_field(ex):
    """One scene whose distance field ends before its d_safe beside one whose
    does not."""
    scenes = _scenes([(300, 20, 2000), (300, 20, 1500)], False, 12)
    scenes[1]["params"]["d_safe"] = 7.0
    dev = [_dev_scene(ex, s) for s in scenes]
    b = ex.Batch(dev, dmin=False)
    b.step()
    _check(ex, scenes, dev, b, True)
