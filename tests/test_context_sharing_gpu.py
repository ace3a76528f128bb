"""What the calls of one context leave behind for each other: nothing."""
import numpy as np
import pytest

import synth

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


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@pytest.mark.parametrize("kind,fp", [(synth.POLYGON, synth.l_footprint()), (synth.RECTS, synth.forklift_rects())])
def test_overlapping_split_calls_leave_nothing_behind(ex, kind, fp):
    """Calls that split a pose over many blocks must not overlap on one context;
    where they do all the same (two streams, different numbers of blocks per
    pose, one of them a replayed graph), a later call that runs alone still gives
    its own minimum: the exact values of the call without a context."""
    import torch
    g = synth.rng(11)
    f, ctx = ex.Footprint(kind, fp), ex.Context()
    poses = _t(g.uniform(-3, 3, (120, 3)))
    clouds = [_t(g.uniform(-6, 6, (n, 2))) for n in (60_000, 6_000, 7_500)]
    outs = [dict(dmin=torch.empty(120, device="cuda"), argmin=torch.empty(120, dtype=torch.int32, device="cuda"))
            for _ in clouds]
    streams = [torch.cuda.Stream() for _ in clouds]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=streams[2]):
        ex.sdf_batch(clouds[2], poses, f, dist=False, ctx=ctx, out=outs[2])
    for _ in range(40):
        for k in (0, 1):
            with torch.cuda.stream(streams[k]):
                ex.sdf_batch(clouds[k], poses, f, dist=False, ctx=ctx, out=outs[k])
        with torch.cuda.stream(streams[2]):
            graph.replay()
    torch.cuda.synchronize()
    for pts in clouds:
        _, m, a = ex.sdf_batch(pts, poses, f, dist=False, ctx=ctx)
        _, m0, a0 = ex.sdf_batch(pts, poses, f, dist=False)
        assert torch.equal(m, m0) and torch.equal(a, a0)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(outs[2]["dmin"], m0) and torch.equal(outs[2]["argmin"], a0)


@pytest.mark.parametrize("P,N", [(1, 513), (3, 1000), (300, 1537), (2, 4095), (160, 30_001), (700, 3000)])
def test_clustered_blocks_of_a_pose_meet(ex, P, N):
    """Two, four and eight blocks per pose, the last of them without points too,
    masked and not, on two streams at once: the exact values of the call
    without a context."""
    import torch
    g = synth.rng(P + N)
    f, ctx = ex.Footprint.polygon(synth.l_footprint()), ex.Context()
    pts, poses, m = _t(g.uniform(-6, 6, (N, 2))), _t(g.uniform(-3, 3, (P, 3))), torch.from_numpy((g.random(N) < 0.5).astype(np.uint8)).cuda()
    want = [ex.sdf_batch(pts, poses, f, mask) for mask in (None, m)]
    torch.cuda.synchronize()
    got, streams = [], [torch.cuda.Stream() for _ in range(2)]
    for mask, s in zip((None, m), streams):
        with torch.cuda.stream(s):
            got += [ex.sdf_batch(pts, poses, f, mask, ctx=ctx) for _ in range(3)]
    torch.cuda.synchronize()
    for k, r in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(r, want[k // 3]))


class _Cycle:
    """A cycle on buffers of its own, from the same nominal every time."""

    def __init__(self, ex, ctx, K, T, N, dmin, seed):
        s = synth.plain_step(seed, K=K, T=T, N=N)
        s["params"] = synth.mppi_params(K, T, synth.OMNI)
        s["eps"], s["U"] = synth.noise(synth.rng(seed), K, T, (0.5, 0.5, 1.0)), np.full((T, 3), 0.2, np.float32)
        self.ex, self.ctx, self.dmin, self.out = ex, ctx, dmin, {}
        self.t = {k: _t(s[k]) for k in ("q0", "cloud", "waypoints", "U", "eps")}
        self.u0, self.fp, self.params = self.t["U"].clone(), ex.Footprint(s["kind"], s["fp"]), s["params"]

    def run(self, ctx=None, out=None):
        t, out = self.t, self.out if out is None else out
        t["U"].copy_(self.u0)
        out.update(self.ex.mppi_step(ctx or self.ctx, t["q0"], t["cloud"], t["waypoints"], t["U"], t["eps"], self.fp,
                                     self.params, dmin=self.dmin, out=out))

    def check(self, what):
        import torch
        torch.cuda.synchronize()
        got, want = {k: v.clone() for k, v in self.out.items()}, {}
        for v in self.out.values():
            v.zero_()
        self.run(self.ex.Context(), want)
        torch.cuda.synchronize()
        for k in want:
            assert torch.equal(got[k], want[k]), (what, k)


@pytest.mark.parametrize("dmin,N", [(False, 300), (True, 2000)])
@pytest.mark.parametrize("a,b", [((64, 10), (128, 20)), ((151, 5), (40, 128)), ((16, 64), (1000, 30)), ((100, 12), (60, 40))])
def test_replays_and_eager_cycles_of_other_sizes_take_turns(ex, a, b, dmin, N):
    """Horizons split over several blocks: a graph replayed between eager cycles
    of other sizes on the same context, and eager cycles of one size with a
    replay of another between them, each give what a fresh context gives."""
    import torch
    ctx = ex.Context()
    ctx.reserve(0, 1000, 128, N)
    A, B = _Cycle(ex, ctx, *a, N, dmin, 1), _Cycle(ex, ctx, *b, N, dmin, 2)
    B.run()
    A.run()   # the usual warm-up before a capture
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        A.run()
    for k in range(3):
        B.run()
        B.check(f"eager {k}")
        graph.replay()
        A.check(f"replay {k}")
        graph.replay()
        B.run()
        A.check(f"replay before eager {k}")
        B.run()
        B.check(f"eager after replay {k}")


@pytest.mark.parametrize("dist,P,N", [(False, 3000, 20_000), (True, 1000, 60_000)])
def test_reserve_holds_what_many_pose_calls_take(ex, dist, P, N):
    """A context reserved for its poses and points makes and maps its memory
    then: the first call takes none from the device."""
    import torch
    g = synth.rng(P)
    f = ex.Footprint.polygon(synth.star_polygon(g, 24, 0.3, 1.2))
    pts, poses = _t(g.uniform(-6, 6, (N, 2))), _t(g.uniform(-3, 3, (P, 3)))
    out = dict(zip(("dist", "dmin", "argmin"), ex.sdf_batch(pts, poses, f, dist=True, ctx=ex.Context())))
    want = {k: v.clone() for k, v in out.items()}
    first = ex.Context()
    ex.sdf_batch(pts, poses, f, dist=dist, ctx=first, out=out)   # loads the kernels
    torch.cuda.synchronize()
    first.close()                                                # and gives its memory back
    ctx = ex.Context()
    ctx.reserve(P, 0, 0, N)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ex.sdf_batch(pts, poses, f, dist=dist, ctx=ctx, out=out)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    assert all(torch.equal(out[k], want[k]) for k in want)


def test_contexts_share_the_pool_and_the_last_gives_it_back(ex):
    """Two contexts' many-pose calls on two streams, one context going while the
    other works on; with the last the memory is the device's again."""
    import gc
    import torch
    gc.collect()
    g = synth.rng(3)
    f = ex.Footprint.polygon(synth.star_polygon(g, 24, 0.3, 1.2))
    N = 2_000_000   # 20 MB of sorted chunks per call
    pts, poses = _t(g.uniform(-6, 6, (N, 2))), _t(g.uniform(-3, 3, (300, 3)))
    want = ex.sdf_batch(pts, poses, f, dist=False)
    ex.sdf_batch(pts, poses, f, dist=False, ctx=ex.Context())   # loads the kernels
    torch.cuda.synchronize()
    gc.collect()
    outs = [dict(dmin=torch.empty(300, device="cuda"), argmin=torch.empty(300, dtype=torch.int32, device="cuda")) for _ in range(2)]
    free = torch.cuda.mem_get_info()[0]
    ctxs, streams = [ex.Context() for _ in outs], [torch.cuda.Stream() for _ in outs]
    for turn in range(3):
        for k in range(2):
            if ctxs[k]:
                with torch.cuda.stream(streams[k]):
                    ex.sdf_batch(pts, poses, f, dist=False, ctx=ctxs[k], out=outs[k])
        torch.cuda.synchronize()
        for o in outs:
            assert torch.equal(o["dmin"], want[1]) and torch.equal(o["argmin"], want[2])
            o["dmin"].zero_() if turn == 0 else None
        if turn == 1:
            ctxs[0].close()
            ctxs[0] = None
    assert free - torch.cuda.mem_get_info()[0] >= 20 << 20
    ctxs[1].close()
    assert free - torch.cuda.mem_get_info()[0] < 4 << 20   # the contexts' own allocations may stay with the driver
