"""The paths that leave out work that cannot matter, against the general ones:
bit for bit, at the sizes and clouds where their cells, runs, queues, patches
and rows end.  The general paths (a d_min output; no context) are themselves
compared with the FP64 oracle elsewhere."""
import numpy as np
import pytest

import synth
from test_mppi_gpu import run_gpu as run_cycle

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


def _cloud(kind, n, g):
    if kind == "uniform":
        return g.uniform(-3, 3, (n, 2))
    if kind == "wall":        # long runs in few cells, straight through the body
        return np.stack([np.linspace(-1, 4, n), np.full(n, 0.1)], 1)
    if kind == "point":       # every point in one cell
        return np.tile([[0.6, 0.05]], (n, 1))
    if kind == "outlier":     # one far point stretches the cells over everything else
        p = g.uniform(-2, 2, (n, 2))
        p[n // 2] = (3.0e5, -2.0e5)
        return p
    p = g.uniform(-3, 3, (n, 2))          # "invalid": non-finite points are as good as masked
    p[::7] = np.nan
    p[1::11, 0] = np.inf
    return p


FOOTPRINTS = {"L": (synth.POLYGON, synth.l_footprint()), "forklift": (synth.RECTS, synth.forklift_rects()),
              "star64": (synth.POLYGON, synth.star_polygon(synth.rng(1), 64, 0.3, 1.0)),
              "far": (synth.POLYGON, synth.l_footprint() + np.float32(2.5))}   # body origin outside the footprint


def _cycle(cloud, n, fp, K, T, model, seed, mask=False):
    g = synth.rng(seed)
    s = dict(synth.plain_step(seed, K=K, T=T, N=8))
    s["cloud"] = _cloud(cloud, n, g).astype(np.float32)
    s["mask"] = (g.random(n) < 0.7).astype(np.uint8) if mask else None
    s["kind"], s["fp"] = FOOTPRINTS[fp]
    s["params"] = synth.mppi_params(K, T, model)
    s["eps"] = synth.noise(g, K, T, {synth.DIFF: (0.5, 1.0), synth.OMNI: (0.5, 0.5, 1.0), synth.SPIN: (1.0,)}[model])
    s["U"] = np.full((T, s["params"]["nu"]), 0.2, np.float32)
    return s


@pytest.mark.parametrize("cloud,n,fp,K,T,model,mask", [
    ("uniform", 1024, "L", 1, 1, synth.DIFF, False), ("uniform", 5000, "forklift", 257, 33, synth.OMNI, True),
    ("uniform", 4096, "star64", 3651, 20, synth.DIFF, False), ("wall", 4097, "forklift", 459, 40, synth.DIFF, False),
    ("wall", 9000, "star64", 40, 128, synth.DIFF, True), ("point", 3000, "L", 130, 24, synth.OMNI, False),
    ("outlier", 2500, "far", 300, 20, synth.SPIN, False), ("invalid", 2048, "L", 912, 10, synth.DIFF, True),
    ("uniform", 30000, "far", 16, 60, synth.DIFF, False), ("uniform", 1500, "L", 7300, 128, synth.DIFF, False),
    ("wall", 1100, "L", 4000, 70, synth.OMNI, False)])
def test_grid_cycle_equals_unpruned_bitwise(ex, cloud, n, fp, K, T, model, mask):
    """Cell grid and distance field against the evaluation of every point (a
    d_min output switches them off): one sample, ragged sample groups, every
    point in one cell, long runs through the footprint, an outlier that
    stretches the cells, non-finite points, a footprint away from its origin."""
    s = _cycle(cloud, n, fp, K, T, model, K + T, mask)
    if cloud == "invalid":   # what non-finite points stand for, for the unpruned run
        bad = ~np.isfinite(s["cloud"]).all(axis=1)
        a_s = dict(s, cloud=np.where(bad[:, None], np.float32(0), s["cloud"]), mask=s["mask"] * ~bad)
    else:
        a_s = s
    a, b = run_cycle(ex, ex.Context(), a_s, dmin=True), run_cycle(ex, ex.Context(), s, dmin=False)
    for k in ("costs", "weights", "U_upd", "U", "u_star"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    assert a["valid"] == b["valid"]


@pytest.mark.parametrize("threads", [64, 128, 512])
def test_grid_batch_any_block_size(ex, threads):
    """Scenes of a batch at every block size (more samples per item than warps
    included), mixed with a scene that has a d_min output in another batch."""
    import torch
    scenes = [_cycle(c, n, fp, K, T, synth.DIFF, 5 + i) for i, (c, n, fp, K, T) in enumerate(
        [("uniform", 700, "L", 67, 20), ("wall", 2500, "forklift", 2000, 25), ("point", 64, "star64", 800, 9),
         ("uniform", 1, "L", 900, 40)])]
    dev = [dict(state=torch.from_numpy(s["q0"]).cuda(), cloud=torch.from_numpy(s["cloud"]).cuda(),
                waypoints=torch.from_numpy(s["waypoints"]).cuda(), U=torch.from_numpy(s["U"]).cuda(),
                noise=torch.from_numpy(s["eps"]).cuda(), fp=ex.Footprint(s["kind"], s["fp"]), params=s["params"])
           for s in scenes]
    b = ex.Batch(dev)
    b.set_tiles(threads, 1)
    b.step()
    torch.cuda.synchronize()
    assert b.get_error() == 0
    for s, o, d in zip(scenes, b.outputs, dev):
        a = run_cycle(ex, ex.Context(), s, dmin=True)
        for k in ("costs", "weights", "U_upd", "u_star"):
            np.testing.assert_array_equal(o[k].cpu().numpy(), a[k], err_msg=k)
        np.testing.assert_array_equal(d["U"].cpu().numpy(), a["U"])


def _poses(g, P, half):
    return np.concatenate([g.uniform(-half, half, (P, 2)), g.uniform(-np.pi, np.pi, (P, 1))], 1).astype(np.float32)


def _both(ex, pts, poses, kind, fp, mask, dist):
    import torch
    f = ex.Footprint(kind, fp)
    args = [torch.from_numpy(a).cuda() for a in (pts, poses)]
    m = None if mask is None else torch.from_numpy(mask).cuda()
    out = []
    for ctx in (None, ex.Context()):   # no scratch, no pruned path
        r = ex.sdf_batch(args[0], args[1], f, m, dist=dist, ctx=ctx)
        torch.cuda.synchronize()
        out.append(r)
    return out


@pytest.mark.parametrize("E,P,N,mask,scale", [
    (12, 3000, 8192, False, 1.0), (31, 1100, 8191, True, 1.0), (32, 1100, 8193, False, 1.0), (33, 520, 16384, False, 1.0),
    (64, 70, 60001, True, 1.0), (64, 40000, 128, False, 1.0), (40, 900, 8192, False, 200.0), (16, 2200, 8188, False, 0.02)])
def test_sdf_matrix_pruned_equals_general_bitwise(ex, E, P, N, mask, scale):
    """Patches, edges left out, rows gathered in shared memory: both word counts
    of the edge mask with and without a padding edge, one patch, ragged and
    several chunks, row lengths that are and are not a multiple of 16 bytes,
    masked and non-finite points, coordinates far beyond and far below the
    footprint's size, a heading of exactly 0."""
    g = synth.rng(E + N)
    pts = (g.uniform(-6, 6, (N, 2)) * scale).astype(np.float32)
    pts[3], pts[7, 1] = np.nan, np.inf
    poses = _poses(g, P, 5 * scale)
    poses[1] = (0.25, -0.5, 0.0)
    m = (g.random(N) < 0.8).astype(np.uint8) if mask else None
    (d0, m0, a0), (d1, m1, a1) = _both(ex, pts, poses, synth.POLYGON, synth.star_polygon(g, E, 0.3, 1.2), m, True)
    assert bool((d0 == d1).all())
    assert bool((m0 == m1).all()) and bool((a0 == a1).all())


@pytest.mark.parametrize("fp,P,N,mask,half", [
    ("star12", 300, 8192, False, 6.0), ("L", 256, 20001, True, 6.0), ("forklift", 5000, 700, False, 6.0),
    ("star64", 400, 8200, True, 500.0), ("L", 20000, 129, False, 1.0)])
def test_sdf_minimum_pruned_equals_general_bitwise(ex, fp, P, N, mask, half):
    """The minimum alone: whole and ragged chunks, duplicated points (the
    lowest index wins a tie), no valid point at all, rectangle covers."""
    g = synth.rng(P + N)
    kind, verts = (synth.POLYGON, synth.star_polygon(g, 12, 0.3, 1.2)) if fp == "star12" else FOOTPRINTS[fp]
    pts = g.uniform(-half, half, (N, 2)).astype(np.float32)
    pts[N // 2:] = pts[:N - N // 2]
    poses = _poses(g, P, half)
    for m in ((g.random(N) < 0.8).astype(np.uint8) if mask else None, np.zeros(N, np.uint8)):
        (_, m0, a0), (_, m1, a1) = _both(ex, pts, poses, kind, verts, m, False)
        assert bool((m0 == m1).all()) and bool((a0 == a1).all())


def test_sdf_under_capture_without_scratch_takes_the_general_path(ex):
    """A capturing stream may not allocate: a context reserved for the poses
    only still captures the call, and the replay gives the same bits."""
    import torch
    g = synth.rng(9)
    pts, poses = torch.from_numpy(g.uniform(-6, 6, (8192, 2)).astype(np.float32)).cuda(), torch.from_numpy(_poses(g, 3000, 5)).cuda()
    f = ex.Footprint.polygon(synth.star_polygon(g, 16, 0.3, 1.2))
    ctx = ex.Context()
    ctx.reserve(3000, 0, 0)
    o = dict(dmin=torch.empty(3000, device="cuda"), argmin=torch.empty(3000, dtype=torch.int32, device="cuda"))
    st, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        ex.sdf_batch(pts, poses, f, dist=False, out=dict(o))   # first-time work, without the context
        st.synchronize()
        with torch.cuda.graph(graph, stream=st):
            ex.sdf_batch(pts, poses, f, dist=False, ctx=ctx, out=o)
    graph.replay()
    torch.cuda.synchronize()
    _, m, a = ex.sdf_batch(pts, poses, f, dist=False, ctx=ex.Context())
    assert bool((o["dmin"] == m).all()) and bool((o["argmin"] == a).all())


@pytest.mark.parametrize("n_cloud,n_pts", [(1500, 200_000), (500, 20_000), (500, 200_000)])
def test_captured_cycle_survives_scratch_growth(ex, n_cloud, n_pts):
    """A graph keeps the scratch it was captured with, and its counters: a later
    call of the same context, with or without a need for more scratch, must not
    take either away."""
    import torch
    s = synth.plain_step(3, K=64, T=10, N=n_cloud)
    dev = torch.device("cuda")
    t = {k: torch.from_numpy(s[k]).to(dev) for k in ("q0", "cloud", "waypoints", "U", "eps")}
    fp = ex.Footprint(s["kind"], s["fp"])
    ctx = ex.Context()
    outs = {}
    u0 = t["U"].clone()

    def cycle(c, out):
        t["U"].copy_(u0)
        out.update(ex.mppi_step(c, t["q0"], t["cloud"], t["waypoints"], t["U"], t["eps"], fp, s["params"], out=out))
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        cycle(ctx, outs)
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        cycle(ctx, outs)
    g = synth.rng(4)
    pts = torch.from_numpy(g.uniform(-6, 6, (n_pts, 2)).astype(np.float32)).to(dev)
    poses = torch.from_numpy(g.uniform(-3, 3, (1000, 3)).astype(np.float32)).to(dev)
    _, grown, _ = ex.sdf_batch(pts, poses, fp, dist=False, ctx=ctx)
    graph.replay()
    torch.cuda.synchronize()
    want = {}
    cycle(ex.Context(), want)
    torch.cuda.synchronize()
    for k in want:
        assert torch.equal(outs[k], want[k]), k
    assert torch.equal(grown, ex.sdf_batch(pts, poses, fp, dist=False)[1])


def test_many_pose_calls_of_one_context_overlap(ex):
    """Calls of many poses on two streams share nothing but the context."""
    import torch
    g = synth.rng(5)
    fp = ex.Footprint(synth.POLYGON, synth.star_polygon(g, 20, 0.3, 1.0))
    ctx = ex.Context()
    sets = [(torch.from_numpy(g.uniform(-6, 6, (20_000, 2)).astype(np.float32)).cuda(),
             torch.from_numpy(g.uniform(-3, 3, (700, 3)).astype(np.float32)).cuda()) for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in sets]
    torch.cuda.synchronize()
    got = []
    for _ in range(4):
        for (pts, poses), s in zip(sets, streams):
            with torch.cuda.stream(s):
                got.append(ex.sdf_batch(pts, poses, fp, dist=True, ctx=ctx))
                got.append(ex.sdf_batch(pts, poses, fp, dist=False, ctx=ctx))
    torch.cuda.synchronize()
    for i, (d, m, a) in enumerate(got):
        want = ex.sdf_batch(*sets[i // 2 % 2], fp)
        assert torch.equal(m, want[1]) and torch.equal(a, want[2])
        assert d is None or torch.equal(d, want[0])
