"""The pruned paths at the ends of their ranges: far from the map's origin, with
points far from all others, with safety distances beyond the scene.  Bit for bit
against the evaluation of every point."""
import numpy as np
import pytest

import synth
from test_mppi_gpu import run_gpu as run_cycle
from test_pruned_paths_gpu import FOOTPRINTS, _both, _cycle, ex  # noqa: F401 (ex: the fixture)

pytestmark = pytest.mark.gpu


def _same_cycle(ex, s):  # noqa: F811
    a, b = run_cycle(ex, ex.Context(), s, dmin=True), run_cycle(ex, ex.Context(), s, dmin=False)
    for k in ("costs", "weights", "U_upd", "U", "u_star"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    assert a["valid"] == b["valid"]


@pytest.mark.parametrize("at", [(1e4, -1e4), (-1e5, 1e5), (5e5, 4.5e6), (3e7, 0.0)])
@pytest.mark.parametrize("cloud,fp,theta", [("uniform", "forklift", 0.0), ("wall", "far", np.pi / 2), ("uniform", "star64", 0.7)])
def test_grid_cycle_in_map_coordinates(ex, at, cloud, fp, theta):  # noqa: F811
    """Where the coordinates' own spacing is 1 mm, 8 mm, 0.5 m and 2 m."""
    s = _cycle(cloud, 3000, fp, 300, 25, synth.DIFF, 77)
    s["cloud"] = (s["cloud"] + np.array(at)).astype(np.float32)
    s["waypoints"] = (s["waypoints"] + np.array(at)).astype(np.float32)
    s["q0"] = np.array([at[0], at[1], theta], np.float32)
    _same_cycle(ex, s)


@pytest.mark.parametrize("at", [(1e4, 1e4), (-2e5, 1e5), (3e7, 0.0)])
@pytest.mark.parametrize("dist", [True, False])
def test_sdf_pruned_in_map_coordinates(ex, at, dist):  # noqa: F811
    g = synth.rng(31)
    pts = (g.uniform(-6, 6, (9000, 2)) + np.array(at)).astype(np.float32)
    poses = np.concatenate([g.uniform(-5, 5, (1500, 2)) + np.array(at), g.uniform(-3, 3, (1500, 1))], 1).astype(np.float32)
    poses[0, 2] = 0.0
    (d0, m0, a0), (d1, m1, a1) = _both(ex, pts, poses, synth.POLYGON, synth.star_polygon(g, 32, 0.3, 1.2), None, dist)
    assert d0 is None or bool((d0 == d1).all())
    assert bool((m0 == m1).all()) and bool((a0 == a1).all())


@pytest.mark.parametrize("N,T,speed", [(120_000, 80, 0.3), (4000, 25, 30.0), (1_200_000, 128, 1.0)])
def test_predicted_cycle_with_a_grid_per_step_or_one(ex, N, T, speed):  # noqa: F811
    """Grids of all steps together below and above 64 MB, and beyond 1 GB (one
    grid for all steps): the bits of the evaluation of every point."""
    import torch
    g = synth.rng(N)
    s = synth.plain_step(4, K=8, T=T, N=8)
    t = {k: torch.from_numpy(np.ascontiguousarray(s[k])).cuda() for k in ("q0", "waypoints", "eps")}
    cloud = torch.from_numpy(g.uniform(-40, 40, (N, 2)).astype(np.float32)).cuda()
    vel = torch.from_numpy(g.normal(0, speed, (N, 2)).astype(np.float32)).cuda()
    fp, res = ex.Footprint(s["kind"], s["fp"]), []
    for dmin in (True, False):
        U = torch.from_numpy(s["U"]).cuda()
        o = ex.mppi_step(ex.Context(), t["q0"], cloud, t["waypoints"], U, t["eps"], fp, s["params"], velocity=vel, dmin=dmin)
        res.append(dict(o, U=U))
    for k in ("costs", "weights", "U_upd", "u_star", "valid", "U"):
        assert torch.equal(res[0][k], res[1][k]), k


@pytest.mark.parametrize("d_safe", [0.0, -1.0, 2.0, 50.0, 3e4, 1e12, 1e25, np.inf])
@pytest.mark.parametrize("cloud,fp,mask", [("uniform", "forklift", True), ("wall", "far", False), ("uniform", "star64", False)])
def test_grid_cycle_at_any_safety_distance(ex, d_safe, cloud, fp, mask):  # noqa: F811
    """The field that ends before d_safe, points inside it, beyond it and none of
    them; distances whose squares overflow (costs that are not numbers, the same
    ones), none and negative ones."""
    s = _cycle(cloud, 2500, fp, 200, 25, synth.DIFF, 3, mask)
    s["params"]["d_safe"] = d_safe
    if d_safe == 50.0:
        s["cloud"] += np.float32(30.0)
    _same_cycle(ex, s)


def _far_points(g, n, half, at, share):
    """A cloud on [-half, half]^2 with a share of its points (at least one) around
    places `at` metres away, in every direction."""
    p = g.uniform(-half, half, (n, 2))
    far = g.permutation(n)[:max(1, int(share * n))]
    a = g.uniform(-np.pi, np.pi, far.size)
    p[far] = np.stack([np.cos(a), np.sin(a)], 1) * at * g.uniform(0.5, 1.0, (far.size, 1))
    return p.astype(np.float32)


@pytest.mark.parametrize("at,share", [(1e3, 0.0), (1e6, 0.0), (1e30, 0.0), (300.0, 0.01), (4e3, 0.05), (4e3, 0.3)])
@pytest.mark.parametrize("n,fp,K,T", [(1024, "forklift", 200, 30), (5000, "far", 150, 128), (9000, "star64", 900, 20)])
def test_grid_cycle_with_points_far_away(ex, at, share, n, fp, K, T):  # noqa: F811
    """Cells laid over the window most points lie in, once and several times, and
    not; rollouts that stay in the window and, at 40 m/s, leave it towards the
    points that its border cells hold."""
    for speed in (0.3, 40.0):
        s = _cycle("uniform", n, fp, K, T, synth.DIFF, K + n)
        s["cloud"] = _far_points(synth.rng(n), n, 4.0, at, share)
        s["U"] = np.tile(np.float32([speed, 0.01]), (T, 1))
        _same_cycle(ex, s)


@pytest.mark.parametrize("speed", [0.5, 50.0])
@pytest.mark.parametrize("N,T", [(3000, 20), (1_200_000, 128)])
def test_predicted_cycle_with_points_far_away(ex, N, T, speed):  # noqa: F811
    """The same for predicted clouds, with a grid per step and with one for all:
    the fastest point may be one of those outside the window."""
    import torch
    g = synth.rng(N)
    s = synth.plain_step(4, K=8, T=T, N=8)
    t = {k: torch.from_numpy(np.ascontiguousarray(s[k])).cuda() for k in ("q0", "waypoints", "eps")}
    p = _far_points(g, N, 6.0, 5e3, 0.001)
    vel = torch.from_numpy(np.where(np.abs(p).max(axis=1, keepdims=True) > 7, -p / 2, g.normal(0, speed, (N, 2))).astype(np.float32)).cuda()
    cloud, fp, res = torch.from_numpy(p).cuda(), ex.Footprint(s["kind"], s["fp"]), []
    for dmin in (True, False):
        U = torch.from_numpy(s["U"]).cuda()
        o = ex.mppi_step(ex.Context(), t["q0"], cloud, t["waypoints"], U, t["eps"], fp, s["params"], velocity=vel, dmin=dmin)
        res.append(dict(o, U=U))
    for k in ("costs", "weights", "U_upd", "u_star", "valid", "U"):
        assert torch.equal(res[0][k], res[1][k]), k


@pytest.mark.parametrize("at,share", [(1e3, 0.0), (1e6, 0.0), (1e30, 0.0), (300.0, 0.01), (4e3, 0.05)])
@pytest.mark.parametrize("N,dist", [(8192, True), (20_003, True), (9001, False), (700, False)])
def test_sdf_pruned_with_points_far_away(ex, at, share, N, dist):  # noqa: F811
    g = synth.rng(N)
    pts = _far_points(g, N, 6.0, at, share)
    pts[5] = np.nan
    poses = np.concatenate([g.uniform(-5, 5, (6000, 2)), g.uniform(-3, 3, (6000, 1))], 1).astype(np.float32)
    (d0, m0, a0), (d1, m1, a1) = _both(ex, pts, poses, synth.POLYGON, synth.star_polygon(g, 32, 0.3, 1.2), None, dist)
    assert d0 is None or bool((d0 == d1).all())
    assert bool((m0 == m1).all()) and bool((a0 == a1).all())


@pytest.mark.parametrize("E,N,P,dist", [(16, 8191, 2100, True), (16, 8192, 2100, True), (24, 5461, 2200, True), (24, 5462, 2200, True),
                                        (32, 4095, 2200, True), (32, 4096, 2200, True), (12, 1023, 11_000, False),
                                        (12, 1024, 11_000, False), (0, 70_000, 767, False), (0, 70_000, 768, False)])
def test_sdf_on_both_sides_of_the_pruned_paths_lines(ex, E, N, P, dist):  # noqa: F811
    """E = 0: the rectangle cover."""
    g = synth.rng(N + P)
    pts = g.uniform(-6, 6, (N, 2)).astype(np.float32)
    poses = np.concatenate([g.uniform(-5, 5, (P, 2)), g.uniform(-3, 3, (P, 1))], 1).astype(np.float32)
    kind, fp = (synth.POLYGON, synth.star_polygon(g, E, 0.3, 1.2)) if E else FOOTPRINTS["forklift"]
    (d0, m0, a0), (d1, m1, a1) = _both(ex, pts, poses, kind, fp, None, dist)
    assert d0 is None or bool((d0 == d1).all())
    assert bool((m0 == m1).all()) and bool((a0 == a1).all())
