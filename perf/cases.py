"""Performance cases: the work a user of the library has it do, through the public Python binding.

Families and their ranges:
  sdf       exact_sdf_batch: 1..16,384 poses x 100..1,000,000 points, polygons of 4..64 vertices or covers of 1..8
            rectangles, with and without a mask, the whole distance matrix with its minimum or the minimum alone
  cycle     one control cycle of one robot: K = 64..4,096 samples, T = 10..100 steps, N = 50..20,000 points, every
            planar motion model, static clouds or clouds with predicted motion, the clearance output at small sizes
  hybrid    one cycle of a robot with three motion modes and its mode selection
  batch     one cycle of 8..64 robots whose footprints, clouds and budgets differ (or with one shared footprint)
  train     an epoch of the proposal network: Adam steps on minibatches, then loss and gradient on a held-out batch
  propose   the proposal network's inference for a group of robots: histogram, features, network, candidates

Control cycles run at a fixed rate on fixed buffers, so a robot's program captures its cycle in a CUDA graph once and
replays it every period: these cases do the same.  The other families are called as they are.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_29663_gb300 as ex

DIFF, ACKERMANN, OMNI, SPIN, PARALLEL = ex.DIFF, ex.ACKERMANN, ex.OMNI, ex.SPIN, ex.PARALLEL
SIGMA = {DIFF: (0.3, 0.6), ACKERMANN: (0.3, 0.2), OMNI: (0.3, 0.3, 0.6), PARALLEL: (0.3,), SPIN: (0.5,)}
MODEL_NAMES = {"diff": DIFF, "ackermann": ACKERMANN, "omni": OMNI}
NBINS, R_MAX, T_NET = 64, 10.0, 20          # proposal network: histogram bins, range, horizon
D_IN, D_OUT = NBINS + 7 + 2 * T_NET, 2 * T_NET


def listed():
    return [
        # one clearance query of a scan against a polygon: the smallest call, latency and launches
        dict(name="sdf_call_1x1000", family="sdf", footprint="L", P=1, N=1000, half=25.0, masked=False, dist=True),
        # the evaluator's own benchmark: a full distance matrix against a 32-vertex polygon
        dict(name="sdf_matrix_star32", family="sdf", footprint="star32", P=16384, N=8192, half=6.0, masked=False,
             dist=True),
        # a rectangle cover, padded clouds and a ragged point count
        dict(name="sdf_matrix_rects_masked", family="sdf", footprint="F_rects", P=4096, N=8191, half=6.0,
             masked=True, dist=True),
        # collision checks of many poses against one map: only the minimum is wanted
        dict(name="sdf_min_star12", family="sdf", footprint="star12", P=3000, N=20001, half=8.0, masked=False,
             dist=False),
        # a small robot's cycle: few samples, a short horizon, a small cloud
        dict(name="cycle_plain", family="cycle", footprint="L", model="diff", scene="open", K=256, T=20, N=512,
             moving=False, dmin=False),
        # the sampling budget the method was published with: many samples, long horizon, 100 points
        dict(name="cycle_paper_budget", family="cycle", footprint="T", model="diff", scene="open", K=1000, T=50,
             N=100, moving=False, dmin=False),
        # a forklift in an aisle: rectangle cover, dense scan
        dict(name="cycle_forklift", family="cycle", footprint="forklift", model="ackermann", scene="aisle", K=2048,
             T=40, N=4096, moving=False, dmin=False),
        # moving obstacles with predicted positions along the horizon
        dict(name="cycle_predicted", family="cycle", footprint="L", model="diff", scene="discs", K=1024, T=20,
             N=2048, moving=True, dmin=False),
        # a platform that chooses among three motion modes every cycle
        dict(name="hybrid_3modes", family="hybrid", K=1024, T=20, N=2048),
        # a simulator or a fleet server: 64 robots, each with its own footprint, cloud and budget
        dict(name="batch_64_scenes", family="batch", scenes=64, shared=False, Kmax=4096, Nmax=20000),
        # training the sampling proposal
        dict(name="train_epoch_8x1024", family="train", hidden=256, B=1024, steps=8),
        # the proposal's inference for a group of robots, before their cycles
        dict(name="propose_256_robots", family="propose", hidden=256, B=256, N=2048),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _footprint_name(rng):
    return rng.choice(["star%d" % _log(rng, 4, 64), "star%d" % _log(rng, 4, 64), "rects%d" % rng.randint(1, 8), "L",
                       "T", "forklift"])


def draw(rng):
    family = rng.choice(["sdf", "sdf", "cycle", "cycle", "cycle", "hybrid", "batch", "train", "propose"])
    if family == "sdf":
        P, N = _log(rng, 1, 16384), _log(rng, 100, 1000000)
        N = max(100, min(N, 134000000 // P))
        return dict(family=family, footprint=_footprint_name(rng), P=P, N=N, half=rng.uniform(3.0, 12.0),
                    masked=rng.random() < 0.3, dist=rng.random() < 0.6)
    if family == "cycle":
        K, T, N = _log(rng, 64, 4096), rng.randint(10, 100), _log(rng, 50, 20000)
        return dict(family=family, footprint=_footprint_name(rng), model=rng.choice(sorted(MODEL_NAMES)),
                    scene=rng.choice(["open", "aisle", "discs", "clutter"]), K=K, T=T, N=N,
                    moving=rng.random() < 0.25, dmin=K * T * N < 100000000 and rng.random() < 0.3)
    if family == "hybrid":
        return dict(family=family, K=_log(rng, 128, 2048), T=rng.randint(10, 60), N=_log(rng, 200, 8000))
    if family == "batch":
        return dict(family=family, scenes=rng.randint(8, 64), shared=rng.random() < 0.5, Kmax=_log(rng, 256, 4096),
                    Nmax=_log(rng, 400, 20000))
    if family == "train":
        return dict(family=family, hidden=rng.choice([128, 256, 256, 320, 512]), B=_log(rng, 128, 2048),
                    steps=rng.randint(4, 8))
    return dict(family=family, hidden=rng.choice([128, 256, 256, 320, 512]), B=_log(rng, 1, 512),
                N=_log(rng, 200, 4096))


# ------------------------------------------------------------------ geometry (numpy, seeded)
def _star(g, n, lo, hi):
    while True:
        a = np.sort(g.uniform(0.0, 2.0 * math.pi, n))
        gap = np.diff(np.append(a, a[0] + 2.0 * math.pi))
        if gap.max() < math.pi and gap.min() > 1e-3:
            break
    r = g.uniform(lo, hi, n)
    return np.stack([r * np.cos(a), r * np.sin(a)], 1)


def _footprint(name, g):
    """(kind, float32 array) of a named footprint."""
    if name == "L":
        return ex.POLYGON, np.float32([(-.5, -.3), (.5, -.3), (.5, 1.1), (.2, 1.1), (.2, .3), (-.5, .3)])
    if name == "T":
        return ex.POLYGON, np.float32([(-.15, -.6), (.15, -.6), (.15, .3), (.6, .3), (.6, .6), (-.6, .6), (-.6, .3),
                                       (-.15, .3)])
    if name == "ranger":
        return ex.POLYGON, np.float32([(-.37, -.25), (.37, -.25), (.37, .25), (.25, .25), (.25, .45), (-.05, .45),
                                       (-.05, .25), (-.37, .25)])
    if name == "F_rects":
        return ex.RECTS, np.float32([(-.35, 0, .15, .6), (-.05, .475, .45, .125), (-.15, .025, .35, .125)])
    if name == "forklift":
        return ex.RECTS, np.float32([(0, 0, .9, .5), (1.5, .35, .6, .075), (1.5, -.35, .6, .075)])
    if name.startswith("star"):
        return ex.POLYGON, _star(g, int(name[4:]), 0.3, 1.2).astype(np.float32)
    n = int(name[5:])   # a body and overlapping boxes on it
    c = g.uniform(-0.5, 0.5, (n, 2))
    c[0] = 0.0
    return ex.RECTS, np.concatenate([c, g.uniform(0.1, 0.6, (n, 2))], 1).astype(np.float32)


def _box(cx, cy, w, h, step):
    p = []
    for x0, y0, x1, y1 in ((-1, -1, 1, -1), (1, -1, 1, 1), (1, 1, -1, 1), (-1, 1, -1, -1)):
        k = max(1, int(round((w if y0 == y1 else h) / step)))
        t = np.arange(k)[:, None] / k
        p.append(np.array([[cx + x0 * w / 2, cy + y0 * h / 2]]) * (1 - t) + np.array([[cx + x1 * w / 2,
                                                                                      cy + y1 * h / 2]]) * t)
    return np.concatenate(p)


def _disc(cx, cy, r, step):
    a = np.arange(max(3, int(round(2 * math.pi * r / step)))) * step / r
    return np.stack([cx + r * np.cos(a), cy + r * np.sin(a)], 1)


def _fit(g, p, v, n):
    """A scan fitted to a budget of n points: a uniform subsample in scan order, or zero padding and a mask."""
    if len(p) >= n:
        i = np.sort(g.choice(len(p), n, replace=False))
        return p[i], v[i], None
    m = np.zeros(n, np.uint8)
    m[:len(p)] = 1
    pad = np.zeros((n - len(p), 2))
    return np.concatenate([p, pad]), np.concatenate([v, pad]), m


def _scene(kind, g, n):
    """(cloud, velocities, mask, goal) of a named scene."""
    if kind == "open":      # points all around, outside a clear disc
        p = np.empty((0, 2))
        while len(p) < n:
            q = g.uniform(-4, 4, (2 * n, 2))
            p = np.concatenate([p, q[np.hypot(q[:, 0], q[:, 1]) >= 1.5]])
        a = g.uniform(-math.pi, math.pi, n)
        return (*_fit(g, p, 0.5 * np.stack([np.cos(a), np.sin(a)], 1)[np.arange(len(p)) % n], n), (5.0, 0.0))
    p, v = [], []

    def add(q, vel=(0.0, 0.0)):
        p.append(q)
        v.append(np.tile(vel, (len(q), 1)))

    if kind == "aisle":     # two walls 1.6 m apart, boxes behind them
        x = np.arange(-2.0, 14.0, 0.01)
        for y in (-0.8, 0.8):
            add(np.stack([x, np.full_like(x, y)], 1) + g.normal(0, 0.02, (len(x), 2)))
        for _ in range(30):
            w, h = g.uniform(0.3, 0.8, 2)
            add(_box(g.uniform(2, 14), g.choice([-1, 1]) * (1.2 + h / 2 + g.uniform(0, 2)), w, h, 0.01))
        goal = (5.0, 0.0)
    elif kind == "discs":   # static boxes and moving discs
        for _ in range(8):
            add(_box(g.uniform(1.5, 6), g.uniform(-2.5, 2.5), g.uniform(0.3, 1), g.uniform(0.3, 1), 0.05))
        for _ in range(40):
            r, a, h = g.uniform(1.5, 10), g.uniform(-math.pi, math.pi), g.uniform(-math.pi, math.pi)
            add(_disc(r * math.cos(a), r * math.sin(a), 0.3, 0.05), (0.5 * math.cos(h), 0.5 * math.sin(h)))
        goal = (6.0, 0.0)
    elif kind == "pocket":  # a corridor with a side pocket, the goal inside it
        x, y = np.arange(-4.0, 4.0, 0.02), np.arange(0.9, 3.2, 0.02)
        xo = x[np.abs(x) > 0.8]
        for q in ((x, np.full_like(x, -0.9)), (xo, np.full_like(xo, 0.9)), (np.full_like(y, -0.8), y),
                  (np.full_like(y, 0.8), y)):
            add(np.stack(q, 1))
        for _ in range(12):
            add(_box(g.uniform(-4, 4), g.choice([-1, 1]) * g.uniform(1.6, 4), *g.uniform(0.2, 0.6, 2), 0.02))
        p = [q + g.normal(0, 0.01, q.shape) for q in p]
        goal = (0.0, 2.6)
    else:                   # clutter: 10 to 60 discs and boxes
        for _ in range(int(g.integers(10, 61))):
            r, a = g.uniform(1.5, 8), g.uniform(-math.pi, math.pi)
            c = (r * math.cos(a), r * math.sin(a))
            add(_disc(*c, g.uniform(0.1, 0.5), 0.02) if g.random() < 0.5 else _box(*c, *g.uniform(0.2, 1, 2), 0.02))
        goal = (g.uniform(3, 6), g.uniform(-2, 2))
    return (*_fit(g, np.concatenate(p), np.concatenate(v), n), goal)


def _params(model, K, T, **over):
    steer = model == ACKERMANN
    p = dict(K=K, T=T, nu=ex.NU[model], model=model, dt=0.1, d_safe=0.05, w_coll=1000.0, w_rep=100.0, w_inf=1.0e4,
             w_goal=1.0, w_term=5.0, w_ctrl=0.01, wheelbase=1.4 if steer else 1.0, clamp=int(steer), state_offset=1,
             u_min=[-1e30, -0.6 if steer else -1e30, -1e30], u_max=[1e30, 0.6 if steer else 1e30, 1e30])
    p["lambda"] = 1.0
    return {**p, **over}


def _hybrid_modes(K, T):
    """(model, noise scales, parameters) of the platform's three modes."""
    return [(m, s, _params(m, K, T, wheelbase=0.5, clamp=1, u_min=[-a for a in u] + [-1e30] * (3 - len(u)),
                           u_max=list(u) + [1e30] * (3 - len(u))))
            for m, s, u in ((ACKERMANN, (0.4, 0.3), (1.5, 0.6)), (PARALLEL, (0.3,), (0.6,)), (SPIN, (0.5,), (1.0,)))]


def _batch_plan(case):
    """(model, footprint name, N, K, T) per scene: the case's own, whatever the inputs."""
    g = np.random.default_rng([case["scenes"], case["Kmax"], case["Nmax"]])
    shared = "star%d" % int(g.integers(4, 17))
    return [(int(g.choice([DIFF, ACKERMANN, OMNI])), shared if case["shared"] else "star%d" % int(g.integers(4, 65)),
             int(round(math.exp(g.uniform(math.log(max(100, case["Nmax"] // 100)), math.log(case["Nmax"]))))),
             int(g.choice([case["Kmax"] // 16, case["Kmax"] // 4, case["Kmax"]])), int(g.integers(20, 51)))
            for _ in range(case["scenes"])]


# ------------------------------------------------------------------ inputs on the GPU
def _dev(a, dtype=torch.float32):
    return torch.as_tensor(np.asarray(a)).to("cuda", dtype).contiguous()


def _scene_inputs(g, tg, fp, cloud, vel, mask, goal, model, sigma, params):
    K, T, nu = params["K"], params["T"], params["nu"]
    return dict(state=torch.zeros(3, device="cuda"), cloud=_dev(cloud), velocity=None if vel is None else _dev(vel),
                mask=None if mask is None else _dev(mask, torch.uint8), waypoints=_dev([goal]),
                U=torch.zeros(T, nu, device="cuda"), params=params, kind=fp[0], verts=fp[1],
                noise=(torch.randn(K, T, nu, device="cuda", generator=tg) * _dev(sigma)).contiguous())


def _make(case, seed):
    """The inputs of a case, as plain tensors and arrays."""
    g = np.random.default_rng([int(seed), 17])
    tg = torch.Generator(device="cuda")
    tg.manual_seed(int(seed))
    rand = lambda *s: torch.rand(*s, device="cuda", generator=tg)  # noqa: E731
    fam = case["family"]
    if fam == "sdf":
        P, N, half = case["P"], case["N"], case["half"]
        kind, verts = _footprint(case["footprint"], g)
        poses = torch.cat([(rand(P, 2) * 2 - 1) * half * 5 / 6, (rand(P, 1) * 2 - 1) * math.pi], 1).contiguous()
        return dict(points=(rand(N, 2) * 2 - 1) * half, poses=poses, kind=kind, verts=verts,
                    mask=(rand(N) < 0.9).to(torch.uint8) if case["masked"] else None)
    if fam == "cycle":
        model = MODEL_NAMES[case["model"]]
        fp = _footprint(case["footprint"], g)
        cloud, vel, mask, goal = _scene(case["scene"], g, case["N"])
        return _scene_inputs(g, tg, fp, cloud, vel if case["moving"] else None, mask, goal, model, SIGMA[model],
                             _params(model, case["K"], case["T"]))
    if fam == "hybrid":
        fp = _footprint("ranger", g)
        cloud, _, mask, goal = _scene("pocket", g, case["N"])
        return [_scene_inputs(g, tg, fp, cloud, None, mask, goal, m, s, p)
                for m, s, p in _hybrid_modes(case["K"], case["T"])]
    if fam == "batch":
        fps, out = {}, []
        for model, name, N, K, T in _batch_plan(case):
            fp = fps.setdefault(name, _footprint(name, g)) if case["shared"] else _footprint(name, g)
            cloud, _, mask, goal = _scene("clutter", g, N)
            out.append(_scene_inputs(g, tg, fp, cloud, None, mask, goal, model, SIGMA[model],
                                     _params(model, K, T, wheelbase=1.0)))
        return out
    H, B = case["hidden"], case["B"]
    net = [(g.uniform(-1, 1, s) / math.sqrt(f)).astype(np.float32)
           for s, f in (((H, D_IN), D_IN), ((H,), D_IN), ((H, H), H), ((H,), H), ((D_OUT, H), H), ((D_OUT,), H))]
    if fam == "train":
        n = (case["steps"] + 1) * B
        x = torch.cat([rand(n, NBINS), torch.randn(n, D_IN - NBINS, device="cuda", generator=tg) * 0.5], 1)
        teach = torch.randn(D_IN, D_OUT, device="cuda", generator=tg) / math.sqrt(D_IN)
        y = 0.3 * torch.tanh(x @ teach) + 0.05 * torch.randn(n, D_OUT, device="cuda", generator=tg)
        return dict(net=net, x=x.contiguous(), y=y.contiguous())
    r, a = 0.3 + 5.7 * rand(B, case["N"]).sqrt(), rand(B, case["N"]) * 2 * math.pi
    poses = torch.cat([(rand(B, 2) * 2 - 1) * 10, (rand(B, 1) * 2 - 1) * math.pi], 1).contiguous()
    return dict(net=net, poses=poses, clouds=(torch.stack([r * a.cos(), r * a.sin()], 2) +
                                              poses[:, None, :2]).contiguous(),
                masks=(rand(B, case["N"]) < 0.8).to(torch.uint8), goals=poses[:, :2] + (rand(B, 2) * 2 - 1) * 6,
                prev=rand(B, 2) * 2 - 1, U=(rand(B, T_NET, 2) * 2 - 1).contiguous())


def _captured(step, reset):
    """`step` run once for its first-time work, then captured in a graph; `reset` puts the state back."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        step()
        s.synchronize()
        with torch.cuda.graph(graph, stream=s):
            step()
    torch.cuda.current_stream().wait_stream(s)
    reset()
    torch.cuda.synchronize()
    return graph


def prepare(case, seed):
    d, fam = _make(case, seed), case["family"]
    if fam == "sdf":
        out = dict(dmin=torch.empty(case["P"], device="cuda"),
                   argmin=torch.empty(case["P"], dtype=torch.int32, device="cuda"))
        if case["dist"]:
            out["dist"] = torch.empty(case["P"], case["N"], device="cuda")
        ctx = ex.Context()
        ctx.reserve(case["P"], 0, 0, case["N"])
        return dict(d, case=case, ctx=ctx, out=out, fp=ex.Footprint(d["kind"], d["verts"]))
    if fam == "cycle":
        ctx, fp, outs = ex.Context(), ex.Footprint(d["kind"], d["verts"]), {}
        ctx.reserve(0, case["K"], case["T"], case["N"])

        def step():
            outs.update(ex.mppi_step(ctx, d["state"], d["cloud"], d["waypoints"], d["U"], d["noise"], fp, d["params"],
                                     mask=d["mask"], velocity=d["velocity"], dmin=case["dmin"], out=outs))

        graph = _captured(step, d["U"].zero_)
        return dict(case=case, keep=(ctx, fp, d), graph=graph, outs=dict(outs, U=d["U"]))
    if fam in ("hybrid", "batch"):
        fps = {}
        for sc in d:
            key = (sc["kind"], sc["verts"].tobytes())
            sc["fp"] = fps[key] if key in fps else fps.setdefault(key, ex.Footprint(sc["kind"], sc["verts"]))
        if fam == "hybrid":
            plan = ex.Hybrid(d, lambda_switch=2.0, cool_max=3)
            outs = dict(u=plan.u, mode=plan.mode_state, Jbar=plan.Jbar, U=[sc["U"] for sc in d],
                        costs=[o["costs"] for o in plan.outputs])
            step = plan.step
        else:
            plan, outs = ex.Batch(d, weights=False, U_upd=False), {}

            def step():   # the fleet's results gathered, as its server reads them
                plan.step()
                outs["costs"] = torch.cat([o["costs"] for o in plan.outputs])
                outs["valid"] = torch.cat([o["valid"] for o in plan.outputs])
                outs["u"] = torch.cat([o["u_star"] for o in plan.outputs])
                outs["U"] = torch.cat([sc["U"].view(-1) for sc in d])

        def reset():
            for sc in d:
                sc["U"].zero_()
            if fam == "hybrid":
                plan.mode_state.copy_(torch.tensor([-1, 0, 0], dtype=torch.int32))

        graph = _captured(step, reset)
        return dict(case=case, keep=(plan, d), graph=graph, outs=outs)
    net = ex.MLP(D_IN, case["hidden"], D_OUT, case["B"])
    net.set_params(np.concatenate([w.reshape(-1) for w in d["net"]]))
    return dict(d, case=case, mlp=net, shapes=None)


def run(s):
    case = s["case"]
    fam = case["family"]
    if fam == "sdf":
        dist, dmin, argmin = ex.sdf_batch(s["points"], s["poses"], s["fp"], s["mask"], dist=case["dist"],
                                          ctx=s["ctx"], out=s["out"])
        return dict(dist=dist, dmin=dmin, argmin=argmin)
    if fam in ("cycle", "hybrid", "batch"):
        s["graph"].replay()
        return s["outs"]
    mlp, B = s["mlp"], case["B"]
    if fam == "train":
        losses = [mlp.train_step(s["x"][k * B:(k + 1) * B], s["y"][k * B:(k + 1) * B], 1e-3)
                  for k in range(case["steps"])]
        val, grads = mlp.loss_grad(s["x"][case["steps"] * B:], s["y"][case["steps"] * B:])
        return dict(losses=losses, val=val, grads=grads)
    hist = ex.polar_hist(s["clouds"], s["poses"], NBINS, R_MAX, masks=s["masks"])
    x = ex.proposal_features(hist, s["poses"], s["goals"], s["prev"], s["U"], R_MAX)
    shift = mlp.forward(x)
    U_prop, U_plain = torch.empty_like(s["U"]), torch.empty_like(s["U"])
    ex.proposal_prepare(s["U"], shift, U_prop, U_plain)
    return dict(hist=hist, x=x, U_prop=U_prop, U_plain=U_plain)


def work(case):
    """Bytes: every input read once, every output written once.  Operations: for each (pose, point) the transform,
    one edge or box and the minimum; for each (sample, step) the rollout, the poses and the cost terms; for the
    network its products (forward, and twice that for the gradients)."""
    fam = case["family"]
    if fam == "sdf":
        P, N = case["P"], case["N"]
        return dict(bytes=8 * N + 12 * P + (4 * P * N if case["dist"] else 0) + 8 * P + (N if case["masked"] else 0),
                    flops=P * N * 25)
    if fam == "cycle":
        K, T, N, nu = case["K"], case["T"], case["N"], ex.NU[MODEL_NAMES[case["model"]]]
        return dict(bytes=4 * K * T * nu + (16 if case["moving"] else 8) * N + 8 * K + 12 * T * nu +
                    (4 * K * T if case["dmin"] else 0), flops=60 * K * T + (25 * K * T * N if case["dmin"] else 0))
    if fam == "hybrid":
        return dict(bytes=4 * case["K"] * case["T"] * 4 + 8 * case["N"], flops=3 * 60 * case["K"] * case["T"])
    if fam == "batch":
        plan = _batch_plan(case)
        return dict(bytes=sum(4 * K * T * ex.NU[m] + 8 * N + 4 * K for m, _, N, K, T in plan),
                    flops=sum(60 * K * T for _, _, _, K, T in plan))
    H, B = case["hidden"], case["B"]
    w = H * D_IN + H * H + H * D_OUT
    if fam == "train":
        n = case["steps"]
        return dict(bytes=4 * (n + 1) * B * (D_IN + D_OUT) + n * 24 * w + 4 * w, flops=6.0 * w * B * (n + 1))
    return dict(bytes=B * case["N"] * 9 + 4 * B * (NBINS + D_IN + 3 * D_OUT) + 4 * w,
                flops=2.0 * w * B + 20.0 * B * case["N"])


# ------------------------------------------------------------------ the same results in 64 bits (plain torch)
def _sdf64(px, py, kind, verts):
    """Signed distance of body-frame points to a polygon or a rectangle cover."""
    v = [[float(c) for c in r] for r in np.asarray(verts, np.float64)]
    if kind == ex.RECTS:
        best = None
        for cx, cy, sx, sy in v:
            ax, ay = (px - cx).abs() - sx, (py - cy).abs() - sy
            d = torch.hypot(ax.clamp(min=0), ay.clamp(min=0)) + torch.maximum(ax, ay).clamp(max=0)
            best = d if best is None else torch.minimum(best, d)
        return best
    best, inside = None, torch.zeros_like(px, dtype=torch.bool)
    for (ax, ay), (bx, by) in zip(v, v[1:] + v[:1]):
        dx, dy, ex_, ey = px - ax, py - ay, bx - ax, by - ay
        t = ((dx * ex_ + dy * ey) / (ex_ * ex_ + ey * ey)).clamp(0, 1)
        q = (dx - t * ex_).square() + (dy - t * ey).square()
        best = q if best is None else torch.minimum(best, q)
        if ey != 0.0:
            inside ^= ((py < ay) != (py < by)) & (px < ax + dy * (ex_ / ey))
    return torch.where(inside, -best.sqrt(), best.sqrt())


def _reach(kind, verts):
    """Radius about the body origin that holds the footprint."""
    v = np.asarray(verts, np.float64)
    c = np.abs(v) if kind == ex.POLYGON else np.abs(v[:, :2]) + v[:, 2:]
    return float(np.hypot(c[:, 0], c[:, 1]).max())


def _rollout64(p, u, q0):
    """Scored states (x, y, theta) and the terminal position of control sequences u (R x T x nu)."""
    dt, m = p["dt"], p["model"]
    z = torch.zeros_like(u[..., 0])
    w = {DIFF: lambda: u[..., 1], ACKERMANN: lambda: u[..., 0] / p["wheelbase"] * torch.tan(u[..., 1]),
         OMNI: lambda: u[..., 2], SPIN: lambda: u[..., 0], PARALLEL: lambda: z}[m]()
    th = q0[2] + torch.cumsum(w * dt, 1)
    old = th - w * dt
    c, s = torch.cos(old), torch.sin(old)
    if m in (DIFF, ACKERMANN):
        vx, vy = u[..., 0] * c, u[..., 0] * s
    elif m == OMNI:
        vx, vy = u[..., 0] * c - u[..., 1] * s, u[..., 0] * s + u[..., 1] * c
    elif m == PARALLEL:
        vx, vy = -u[..., 0] * s, u[..., 0] * c
    else:
        vx = vy = z
    return q0[0] + torch.cumsum(vx * dt, 1), q0[1] + torch.cumsum(vy * dt, 1), th


def _clear64(sc, x, y, th, full):
    """Smallest signed distance per scored state (R x T); unless `full`, only what lies within d_safe of the
    footprint matters (every cost is the same beyond) and the rest is +inf."""
    p = sc["params"]
    R, T = x.shape
    keep = slice(None) if sc["mask"] is None else sc["mask"].bool()
    pts = sc["cloud"].double()[keep]
    vel = None if sc["velocity"] is None else sc["velocity"].double()[keep]
    out = torch.full((R * T,), math.inf, dtype=torch.float64, device="cuda")
    if not len(pts):
        return out.view(R, T)
    xs, ys, ths = x.reshape(-1), y.reshape(-1), th.reshape(-1)
    tt = ((torch.arange(T, device="cuda", dtype=torch.float64) + 1) * p["dt"]).repeat(R)
    far = math.inf if full else _reach(sc["kind"], sc["verts"]) + p["d_safe"] + 1e-6
    n = max(1, 30000000 // len(pts))
    for a in range(0, R * T, n):
        b = min(R * T, a + n)
        dx, dy = pts[None, :, 0] - xs[a:b, None], pts[None, :, 1] - ys[a:b, None]
        if vel is not None:
            dx, dy = dx + tt[a:b, None] * vel[None, :, 0], dy + tt[a:b, None] * vel[None, :, 1]
        k = (dx * dx + dy * dy < far * far).nonzero(as_tuple=True)
        c, s, dx, dy = torch.cos(ths[a:b])[k[0]], torch.sin(ths[a:b])[k[0]], dx[k], dy[k]
        d = _sdf64(c * dx + s * dy, c * dy - s * dx, sc["kind"], sc["verts"])
        out[a:b] = out[a:b].scatter_reduce(0, k[0], d, "amin")
    return out.view(R, T)


def _score64(sc, u, full=False):
    """(J, unsafe, clearance) of control sequences u."""
    p, q0 = sc["params"], sc["state"].double()
    x, y, th = _rollout64(p, u, q0)
    d = _clear64(sc, x, y, th, full)
    goal = sc["waypoints"].double()[0]
    dist = torch.hypot(x - goal[0], y - goal[1])
    J = (p["w_goal"] * dist + p["w_ctrl"] * u.square().sum(2) + p["w_coll"] * (d < 0) +
         p["w_rep"] * (p["d_safe"] - d).clamp(min=0).square()).sum(1) + p["w_term"] * dist[:, -1]
    return J, (d < p["d_safe"]).any(1), d


def _cycle64(sc, full=False):
    p, U, nu = sc["params"], sc["U"].double(), sc["params"]["nu"]

    def clip(u):
        if not p["clamp"]:
            return u
        lo, hi = (torch.tensor(p[k][:nu], dtype=torch.float32, device="cuda").double() for k in ("u_min", "u_max"))
        return torch.maximum(torch.minimum(u, hi), lo)

    u = clip(U + sc["noise"].double())
    J, unsafe, d = _score64(sc, u, full)
    costs = J + p["w_inf"] * unsafe
    w = torch.softmax(-(costs - costs.min()) / p["lambda"], 0)
    upd = U + (w[:, None, None] * (u - U)).sum(0)
    Jn, bad, _ = _score64(sc, clip(upd)[None])
    ok = not bool(bad[0])
    new = torch.cat([upd[1:], upd[-1:]]) if ok else torch.zeros_like(upd)
    return dict(costs=costs, weights=w, U_upd=upd, U=new, u_star=upd[0] if ok else torch.zeros_like(upd[0]), dmin=d,
                J=Jn[0], ok=ok)


def _net64(net, x):
    W1, b1, W2, b2, W3, b3 = net
    g = torch.nn.functional.gelu
    return g(g(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3


def exact(case, seed):
    d, fam = _make(case, seed), case["family"]
    if fam == "sdf":
        P, N = case["P"], case["N"]
        dist = torch.empty(P, N, dtype=torch.float64, device="cuda") if case["dist"] else None
        dmin = torch.empty(P, dtype=torch.float64, device="cuda")
        pts, n = d["points"].double(), max(1, 8000000 // N)
        for a in range(0, P, n):
            q = d["poses"][a:a + n].double()
            c, s = torch.cos(q[:, 2:]), torch.sin(q[:, 2:])
            dx, dy = pts[None, :, 0] - q[:, :1], pts[None, :, 1] - q[:, 1:2]
            r = _sdf64(c * dx + s * dy, c * dy - s * dx, d["kind"], d["verts"])
            if d["mask"] is not None:
                r = r.masked_fill(d["mask"][None] == 0, math.inf)
            dmin[a:a + n] = r.amin(1)
            if dist is not None:
                dist[a:a + n] = r
        return dict(dist=dist, dmin=dmin, argmin=None)
    if fam == "cycle":
        r = _cycle64(d, case["dmin"])
        out = {k: r[k] for k in ("u_star", "costs", "weights", "U_upd", "U")}
        return dict(out, valid=None, **({"dmin": r["dmin"]} if case["dmin"] else {}))
    if fam == "hybrid":
        r = [_cycle64(sc) for sc in d]
        J = torch.stack([m["J"] + 2.0 if m["ok"] else m["J"] * 0 + math.inf for m in r])   # no mode yet: all pay
        u, best = torch.zeros(3, dtype=torch.float64, device="cuda"), int(J.argmin())
        if math.isfinite(float(J[best])):
            u[:len(r[best]["u_star"])] = r[best]["u_star"]
        return dict(u=u, mode=None, Jbar=J, U=[m["U"] for m in r], costs=[m["costs"] for m in r])
    if fam == "batch":
        r = [_cycle64(sc) for sc in d]
        return dict(costs=torch.cat([m["costs"] for m in r]), valid=None, u=torch.cat([m["u_star"] for m in r]),
                    U=torch.cat([m["U"].reshape(-1) for m in r]))
    net = [torch.as_tensor(w).to("cuda", torch.float64) for w in d["net"]]
    if fam == "train":
        B, n = case["B"], case["steps"]
        net = [w.requires_grad_() for w in net]
        m, v, losses = [w.detach() * 0 for w in net], [w.detach() * 0 for w in net], []
        for k in range(n + 1):
            x, y = d["x"][k * B:(k + 1) * B].double(), d["y"][k * B:(k + 1) * B].double()
            loss = (_net64(net, x) - y).square().mean()
            grads = torch.autograd.grad(loss, net)
            losses.append(loss.detach().reshape(1))
            if k < n:
                with torch.no_grad():
                    for w, g, a, b in zip(net, grads, m, v):
                        a.mul_(0.9).add_(g, alpha=0.1)
                        b.mul_(0.999).addcmul_(g, g, value=0.001)
                        w -= 1e-3 * (a / (1 - 0.9 ** (k + 1))) / ((b / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
        return dict(losses=losses[:-1], val=losses[-1], grads=torch.cat([g.reshape(-1) for g in grads]))
    q = d["poses"].double()
    c, s = torch.cos(q[:, 2]), torch.sin(q[:, 2])

    def body(o):
        dx, dy = o[..., 0] - q[:, 0].view(-1, *[1] * (o.dim() - 2)), o[..., 1] - q[:, 1].view(-1, *[1] * (o.dim() - 2))
        cc, ss = c.view(-1, *[1] * (o.dim() - 2)), s.view(-1, *[1] * (o.dim() - 2))
        return cc * dx + ss * dy, cc * dy - ss * dx

    px, py = body(d["clouds"].double())
    k = ((torch.atan2(py, px) + math.pi) / (2 * math.pi) * NBINS).floor().long().clamp(0, NBINS - 1)
    r = torch.hypot(px, py).masked_fill(d["masks"] == 0, R_MAX)
    hist = torch.full((len(q), NBINS), R_MAX, dtype=torch.float64, device="cuda").scatter_reduce(1, k, r, "amin")
    gx, gy = body(d["goals"].double())
    dist, U = torch.hypot(gx, gy), d["U"].double()
    x = torch.cat([hist / R_MAX, torch.stack([gx / R_MAX, gy / R_MAX], 1), d["prev"].double(),
                   torch.stack([dist / R_MAX, gx / dist, gy / dist], 1), U.reshape(len(q), -1)], 1)
    return dict(hist=hist, x=x, U_prop=U + _net64(net, x).view_as(U), U_plain=U)
