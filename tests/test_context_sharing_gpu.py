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
