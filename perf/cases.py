"""Performance cases of the planning framework: what a program that plans with it
has it do, through the public entry points of ``paper_2509_17340_gb300.aero``.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` makes the inputs and the handles a program keeps,
``run(state)`` is one pass, ``work(case)`` the bytes and operations it cannot do
without, ``exact(case, seed)`` the same outputs in 64 bits with plain torch.

Kinds of case:
  step    one planning step (``Planner.plan_step``, ``plan_step_host`` or
          ``plan_step_noalloc``): cloud -> partition -> anchors and guides ->
          MPPI ensemble -> update (refined or not) -> Stage II -> selection
  flight  one cycle of the receding-horizon loop: a LiDAR sweep pushed into the
          accumulator, a step on the ring (or on the gathered cloud), the warm
          start shifted
  batch   many planners of uneven sizes in one call (``Batch.plan``)
  grad    cost and gradient of a set of control sequences (``RolloutCost``,
          forward and backward) in the context of a planned step
Every pass starts from the same warm start, so passes on one state are alike.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_17340_gb300 import aero, inputs

DEV = "cuda"
HOVER = [inputs.G, 0.0, 0.0, 0.0]
FLOPS_STEP = 345.0        # FP32 operations of one sample-step: noise, RK4, costs, weighted sum
FLOPS_STAGE2 = 320.0      # of one noise-free step with its costs
FLOPS_GRAD = 960.0        # of one noise-free step forward and backward
BATCH_GRID = {4: (2, 2), 8: (4, 2), 16: (4, 4)}

# Partition geometries of the workloads: fine cones and pooling.
PARTITIONS = {
    "paper": dict(fine_az=120, fine_el=60, pool_az=6, pool_el=6),      # Sec. IV-A, 3 degree cones
    "flight": dict(fine_az=120, fine_el=60, pool_az=6, pool_el=5),     # the closed loop's rows
    "sweep": dict(fine_az=128, fine_el=64, pool_az=8, pool_el=16),     # the ensemble workload
    "large": dict(fine_az=256, fine_el=64, pool_az=4, pool_el=8),      # the large clutter
}


def _step(name, **kw):
    c = dict(name=name, kind="step", entry="device", scene="forest", n=20816, M_h=4, M_v=2, K=1024,
             T=40, dt=0.05, lam=1.0, part="sweep", r_max=10.0, bounds="wide", raw=False, refine=0,
             iters=1, tilted=False, moving_goal=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one MPPI instance without anchors, an onboard rate of a kHz or more
        _step("plain", scene="pillars", n=2000, M_h=1, M_v=1, K=256, T=20, part="paper"),
        # the paper's own settings (Table I, 5 x 3 anchors) on ten accumulated frames
        _step("table1", n=200000, M_h=5, M_v=3, K=128, T=25, lam=0.1, part="paper", bounds="paper"),
        # the ordinary ensemble step on one LiDAR sweep
        _step("ensemble"),
        # the same sizes with five gradient steps on every updated nominal
        _step("refined", scene="pillars", n=2000, refine=5),
        # odd sizes, a tilted start, a moving goal and two MPPI iterations, from a caller that
        # must not allocate
        _step("odd_noalloc", entry="noalloc", n=17321, M_h=3, M_v=1, K=777, T=33, tilted=True,
              moving_goal=True, iters=2),
        # one cycle of the receding-horizon loop
        dict(name="flight", kind="flight", n=15001, frames=10, M_h=4, M_v=2, K=512, T=30, dt=0.05,
             gather=False),
        # the headline step: a dense clutter planned with the whole GPU
        _step("large", scene="clutter", n=200000, M_h=8, M_v=4, K=8192, T=64, dt=0.03, part="large",
              r_max=20.0),
        # the same from and to (page-locked) host memory, as a flight stack on the CPU calls it
        _step("large_host", entry="host", scene="clutter", n=200000, M_h=8, M_v=4, K=8192, T=64,
              dt=0.03, part="large", r_max=20.0),
        # every kept point as the collision set
        _step("large_raw", scene="clutter", n=200000, M_h=8, M_v=4, K=8192, T=64, dt=0.03,
              part="large", r_max=20.0, raw=True),
        # a fleet: 64 planners of uneven sizes in one call
        dict(name="fleet", kind="batch", planners=64, sizes=1),
        # an optimiser's inner loop: 2048 sequences of the ensemble step, cost and gradient
        dict(name="gradient", kind="grad", n=20816, seqs=2048, T=40, dt=0.05),
        # a dense map as the cloud: ten million points into an ordinary step
        _step("dense_map", scene="uniform", n=10_000_000, part="large", r_max=20.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["flight", "batch", "grad"])
    if kind == "flight":
        return dict(kind="flight", n=_log_int(rng, 2000, 18432), frames=rng.randint(2, 16),
                    M_h=rng.randint(1, 6), M_v=rng.randint(1, 3), K=_log_int(rng, 100, 2000),
                    T=rng.randint(15, 60), dt=0.05, gather=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind="batch", planners=_log_int(rng, 2, 64), sizes=rng.randint(2, 1 << 20))
    if kind == "grad":
        return dict(kind="grad", n=_log_int(rng, 2000, 100000), seqs=_log_int(rng, 1, 4000),
                    T=rng.randint(5, 80), dt=0.05)
    c = _step("")
    del c["name"]
    entry = rng.choice(["device", "device", "device", "host", "noalloc"])
    raw = entry != "noalloc" and rng.random() < 0.2
    M_h, M_v = rng.randint(1, 8), rng.randint(1, 4)
    K = _log_int(rng, 64, 8192)
    T = rng.randint(8, 80)
    n = _log_int(rng, 1000, 1_000_000)
    part = rng.choice(["paper", "sweep", "large"])
    scene = rng.choice(["pillars", "forest", "clutter", "uniform"])
    if raw:
        n = min(n, 100_000)
    if entry == "noalloc":
        M_h, M_v, K, T, n = min(M_h, 5), min(M_v, 3), min(K, 2000), min(T, 64), min(n, 65000)
        part = "paper" if part == "large" else part
    K = min(K, (32 * 8192 * 64) // (M_h * M_v * T))
    paper = rng.random() < 0.25
    c.update(entry=entry, raw=raw, scene=scene, n=n, M_h=M_h, M_v=M_v, K=K, T=T, part=part,
             dt=rng.choice([0.03, 0.05]), lam=0.1 if paper else 1.0, bounds="paper" if paper else "wide",
             r_max=rng.choice([10.0, 20.0]), refine=rng.choice([0, 0, 0, 1, 5]),
             iters=rng.choice([1, 1, 1, 2, 3]) if K * M_h * M_v <= 65536 else 1,
             tilted=rng.random() < 0.5, moving_goal=rng.random() < 0.3)
    return c


# ---------------------------------------------------------------------------
# Inputs: parameters and synthetic scenes (drawn on the GPU from the seed)
# ---------------------------------------------------------------------------

def _params(c, seed):
    p = inputs.default_params()
    if c["bounds"] == "wide":  # the benchmark workloads' noise and control bounds
        p.update(sigma=[2.0, 1.5, 1.5, 1.5], u_min=[0.0, -6.0, -6.0, -6.0],
                 u_max=[2 * inputs.G, 6.0, 6.0, 6.0])
    p.update(PARTITIONS[c["part"]])
    p.update(E=c["M_h"] * c["M_v"], M_h=c["M_h"], M_v=c["M_v"], K=c["K"], T=c["T"], dt=c["dt"],
             lam=c["lam"], r_max=c["r_max"], collision_set=int(c["raw"]), iters=c["iters"],
             refine_steps=c["refine"], refine_step=0.05, seed=seed, step_id=seed % 1000)
    if c["M_h"] * c["M_v"] == 1:
        p["Q_track"] = 0.0  # plain MPPI
    if c.get("Q_c") is not None:
        p["Q_c"] = c["Q_c"]
    return p


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV)


def _cylinders(rng, count, half, r_lo, r_hi, h, centre, clear):
    """`count` vertical cylinders (x, y, r, h), none within 2 m of a point of `clear`."""
    c = np.stack([rng.uniform(centre[0] - half, centre[0] + half, 8 * count),
                  rng.uniform(centre[1] - half, centre[1] + half, 8 * count),
                  rng.uniform(r_lo, r_hi, 8 * count), np.full(8 * count, h)], 1)
    for x, y in clear:
        c = c[np.hypot(c[:, 0] - x, c[:, 1] - y) > c[:, 2] + 2.0]
    return torch.from_numpy(c[:count]).float().to(DEV)


def _cast(o, d, cyl, boxes, far):
    """Range of each ray from o along d (R x 3) to the cylinders, boxes and the ground."""
    o = torch.tensor(o, device=DEV)
    t = torch.where(d[:, 2] < 0, -o[2] / d[:, 2], torch.full_like(d[:, 2], 1e9))
    for s in range(0, len(d), 1 << 16):
        e = d[s:s + (1 << 16)]
        a = e[:, 0] ** 2 + e[:, 1] ** 2
        ox, oy = o[0] - cyl[:, 0], o[1] - cyl[:, 1]
        b = e[:, :1] * ox + e[:, 1:2] * oy
        disc = b * b - a[:, None] * (ox * ox + oy * oy - cyl[:, 2] ** 2)
        tt = (-b - disc.clamp_min(0).sqrt()) / a[:, None]
        z = o[2] + tt * e[:, 2:3]
        ok = (disc > 0) & (tt > 0.05) & (z > 0) & (z < cyl[:, 3])
        t[s:s + (1 << 16)] = torch.minimum(t[s:s + (1 << 16)], tt.masked_fill(~ok, 1e9).amin(1))
    for lo, hi in boxes:
        t0, t1 = (torch.tensor(lo, device=DEV) - o) / d, (torch.tensor(hi, device=DEV) - o) / d
        near, off = torch.minimum(t0, t1).amax(1), torch.maximum(t0, t1).amin(1)
        t = torch.where((off >= near) & (near > 0.05), torch.minimum(t, near), t)
    return torch.where(t < far, t, torch.full_like(t, math.nan))


def _sweep(g, o, n_az, n_el, el_lo, el_hi, far, cyl, boxes):
    """One LiDAR sweep from o: hit points (world) with 2 cm range noise."""
    az = torch.arange(n_az, device=DEV) * (2 * math.pi / n_az)
    el = torch.deg2rad(torch.linspace(el_lo, el_hi, n_el, device=DEV))
    A, B = torch.meshgrid(az, el, indexing="ij")
    d = torch.stack([B.cos() * A.cos(), B.cos() * A.sin(), B.sin()], -1).reshape(-1, 3)
    t = _cast(o, d, cyl, boxes, far)
    t = t + 0.02 * torch.randn(t.shape, generator=g, device=DEV)
    p = torch.tensor(o, device=DEV) + t[:, None] * d
    return p[torch.isfinite(t)]


def _pick(g, pts, n):
    """Exactly n of the points."""
    return pts[torch.randint(len(pts), (n,), generator=g, device=DEV)].contiguous()


def _scene(kind, n, seed):
    """(cloud n x 3 float32 on the GPU, start p0, goal)."""
    g, rng = _gen(seed), np.random.default_rng(seed)
    if kind == "pillars":       # surface samples of ten pillars
        cyl = _cylinders(rng, 10, 10.0, 0.2, 0.5, 5.0, (10.0, 0.0), [(0, 0), (18, 0)])
        k = torch.arange(n, device=DEV) % 10
        th, z = _uniform(g, 0, 2 * math.pi, n), _uniform(g, 0, 5, n)
        pts = torch.stack([cyl[k, 0] + cyl[k, 2] * th.cos(), cyl[k, 1] + cyl[k, 2] * th.sin(), z], 1)
        return pts.contiguous(), (0.0, 0.0, 1.5), (18.0, 0.0, 1.5)
    if kind == "forest":        # one sweep in a forest with ground
        cyl = _cylinders(rng, 60, 20.0, 0.2, 0.5, 6.0, (0.0, 0.0), [(0, 0), (18, 0)])
        pts = _sweep(g, (0.0, 0.0, 1.5), 1024, 32, -15.0, 15.0, 30.0, cyl, [])
        if n > len(pts):        # accumulated sweeps, a little apart
            more = [_sweep(g, (0.1 * i, 0.0, 1.5), 1024, 32, -15.0, 15.0, 30.0, cyl, [])
                    for i in range(1, min(10, -(-n // len(pts))))]
            pts = torch.cat([pts] + more)
        return _pick(g, pts, n), (0.0, 0.0, 1.5), (18.0, 0.0, 1.5)
    if kind == "clutter":       # three merged sweeps among thin pillars, wall slabs and ground
        cyl = _cylinders(rng, 300, 30.0, 0.1, 0.3, 10.0, (20.0, 0.0), [(0, 0), (3, 0), (6, 0)])
        boxes = []
        for _ in range(8):
            x, y, w, h = rng.uniform(12, 48), rng.uniform(-25, 25), rng.uniform(4, 8), rng.uniform(3, 8)
            a, b = (0.15, w / 2) if rng.uniform() < 0.5 else (w / 2, 0.15)
            boxes.append(((x - a, y - b, 0.0), (x + a, y + b, h)))
        pts = torch.cat([_sweep(g, (x, 0.0, 2.0), 1800, 64, -30.0, 30.0, 40.0, cyl, boxes)
                         for x in (0.0, 3.0, 6.0)])
        return _pick(g, pts, n), (6.0, 0.0, 2.0), (56.0, 0.0, 2.0)
    # a dense map: uniform points outside a corridor of 3 m around the flight line
    pts = _uniform(g, -20.0, 20.0, n, 3)
    off = (pts[:, 1] ** 2 + pts[:, 2] ** 2).sqrt()
    push = torch.where(off < 3.0, 3.0 / off.clamp_min(1e-3), torch.ones_like(off))
    pts[:, 1:] *= push[:, None]
    pts[:, 2] += 2.0
    return pts.contiguous(), (0.0, 0.0, 2.0), (18.0, 0.0, 2.0)


def _start(c, seed, p0, goal):
    """State (p, q, v) and goal as float32 values, drawn from the seed."""
    rng = np.random.default_rng([seed, 7])
    p = np.array(p0) + rng.uniform(-0.3, 0.3, 3)
    q = np.array([1.0, 0.0, 0.0, 0.0])
    if c.get("tilted"):
        q = q + np.append(0.0, rng.uniform(-0.3, 0.3, 3))
        q /= np.linalg.norm(q)
    fast = c.get("scene") == "clutter"
    v = np.array([rng.uniform(7, 10) if fast else rng.uniform(0, 3), rng.uniform(-0.5, 0.5), 0.0])
    goal = np.array(goal) + rng.uniform(-1.0, 1.0, 3) * [0, 1, 0]
    return tuple(a.astype(np.float32) for a in (p, q, v, goal))


def _warm(P, seed):
    """A warm start: hover with a different small command on every instance."""
    rng = np.random.default_rng([seed, 8])
    u = np.tile(np.array(HOVER, np.float32), (P["E"], P["T"], 1))
    u += rng.normal(0.0, 0.2, (P["E"], 1, 4)).astype(np.float32)
    return torch.from_numpy(u)


def _goal_motion(c, P, seed):
    if c.get("moving_goal"):
        rng = np.random.default_rng([seed, 9])
        q = np.array([1.0, 0, 0, 0]) + np.append(0.0, rng.uniform(-0.2, 0.2, 3))
        P.update(v_goal=[float(x) for x in rng.uniform(-1, 1, 3)],
                 q_goal=[float(x) for x in q / np.linalg.norm(q)])


def _outputs(P):
    return (torch.empty((P["T"], 4), device=DEV), torch.empty((P["E"],), device=DEV),
            torch.empty((1,), dtype=torch.int32, device=DEV))


def _step_inputs(c, seed):
    cloud, p0, goal = _scene(c["scene"], c["n"], seed)
    P = _params(c, seed)
    _goal_motion(c, P, seed)
    p, q, v, goal = _start(c, seed, p0, goal)
    return P, cloud, p, q, v, goal, _warm(P, seed)


def _as_step(c):
    """The step a flight cycle or a gradient case plans."""
    if c["kind"] == "flight":
        return _step("", n=c["n"] * c["frames"], M_h=c["M_h"], M_v=c["M_v"], K=c["K"], T=c["T"],
                     dt=c["dt"], part="flight", Q_c=0.02)
    return _step("", n=c["n"], T=c["T"], dt=c["dt"], K=256)


def _flight_inputs(c, seed):
    """The step's inputs with the frames (sensor points and poses) in place of the cloud."""
    s = _as_step(c)
    P = _params(s, seed)
    g, rng = _gen(seed), np.random.default_rng(seed)
    cyl = _cylinders(rng, 60, 20.0, 0.2, 0.5, 6.0, (0.0, 0.0), [(0, 0), (18, 0)])
    frames = []
    for i in range(c["frames"]):
        o = (0.1 * (i + 1 - c["frames"]), 0.0, 1.5)
        w = _pick(g, _sweep(g, o, 512, 36, -60.0, 30.0, 30.0, cyl, []), c["n"])
        yaw = rng.uniform(-0.3, 0.3)
        q = np.array([math.cos(yaw / 2), 0.0, 0.0, math.sin(yaw / 2)], np.float32)
        R = torch.from_numpy(_rot32(q)).to(DEV)
        frames.append((((w - torch.tensor(o, device=DEV)) @ R).contiguous(), np.array(o, np.float32), q))
    p, q, v, goal = _start(s, seed, (0.0, 0.0, 1.5), (18.0, 0.0, 1.5))
    return P, frames, p, q, v, goal, _warm(P, seed)


def _batch_items(c):
    """The planners' sizes: E in {4, 8, 16}, K in {256, 1024, 4096}, T in {20, 40, 60},
    5,000 to 100,000 points, forest or clutter."""
    rng = np.random.default_rng(c["sizes"])
    out = []
    for i in range(c["planners"]):
        E = int(rng.choice([4, 8, 16]))
        out.append(_step("", scene=["forest", "clutter", "pillars"][int(rng.integers(3))],
                         n=int(np.exp(rng.uniform(np.log(5000), np.log(100000)))),
                         M_h=BATCH_GRID[E][0], M_v=BATCH_GRID[E][1], K=int(rng.choice([256, 1024, 4096])),
                         T=int(rng.choice([20, 40, 60]))))
    return out


def _sequences(c, P, u0, instance, seed):
    """Control sequences around the instance's warm start."""
    g = _gen(seed + 5)
    u = u0[instance].to(DEV) + 0.5 * torch.randn((c["seqs"], c["T"], 4), generator=g, device=DEV)
    lo, hi = (torch.tensor(P[k], device=DEV) for k in ("u_min", "u_max"))
    return torch.minimum(torch.maximum(u, lo), hi).contiguous()


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _planner(P, n):
    return aero.Planner(E_max=P["E"], K_max=P["K"], T_max=P["T"],
                        fine_cells_max=P["fine_az"] * P["fine_el"], n_points_max=n,
                        raw_points_max=0 if P["collision_set"] else -1)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        items, keep = [], []
        steps = _batch_items(case)
        for i, s in enumerate(steps):
            P, cloud, p, q, v, goal, u0 = _step_inputs(s, seed * 64 + i)
            un, outs = u0.to(DEV), _outputs(P)
            items.append(aero.Batch.item(aero.state_struct(p, q, v), cloud, goal, aero.params_struct(P),
                                         un, *outs))
            keep.append((cloud, un, *outs))
        # the warm starts as one buffer each way: one copy resets them all
        flat0 = torch.cat([k[1].reshape(-1) for k in keep])
        flat, at = torch.empty_like(flat0), 0
        for it, k in zip(items, keep):
            it.u_nom_inout = flat.data_ptr() + 4 * at
            at += k[1].numel()
        b = aero.Batch(len(items), E_max=16, K_max=4096, T_max=60, fine_cells_max=128 * 64,
                       n_points_max=max(s["n"] for s in steps))
        return dict(kind=kind, batch=b, items=items, keep=keep, u0=flat0, u=flat)
    if kind == "flight":
        P, frames, p, q, v, goal, u0 = _flight_inputs(case, seed)
        acc = aero.Accumulator(case["frames"], 512 * 36)
        for f in frames:
            acc.push(*f)
        total = case["frames"] * 512 * 36
        u0 = u0.to(DEV)
        return dict(kind=kind, planner=_planner(P, total), acc=acc, frames=frames, at=0,
                    cloud=torch.empty((total, 3), device=DEV) if case["gather"] else None,
                    x=aero.state_struct(p, q, v), goal=goal, P=aero.params_struct(P), u0=u0,
                    u=u0.clone(), scratch=torch.empty_like(u0), outs=_outputs(P),
                    shift=max(1, round(0.1 / case["dt"])))
    s = case if kind == "step" else _as_step(case)
    P, cloud, p, q, v, goal, u0 = _step_inputs(s, seed)
    st = dict(kind=kind, x=aero.state_struct(p, q, v), goal=goal, P=aero.params_struct(P))
    if kind == "step" and s["entry"] == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        st.update(entry="host", planner=_planner(P, s["n"]), cloud=pin(cloud), u0=u0, u=pin(u0),
                  outs=tuple(pin(t) for t in _outputs(P)))
        return st
    u0 = u0.to(DEV)
    st.update(cloud=cloud, u0=u0, u=u0.clone(), outs=_outputs(P))
    if kind == "step":
        st["entry"] = s["entry"]
        if s["entry"] == "device":
            st["planner"] = _planner(P, s["n"])
        return st
    st["planner"] = _planner(P, s["n"])
    st["instance"] = P["E"] // 2
    st["planner"].plan_step(st["x"], cloud, goal, st["P"], st["u"], *st["outs"])
    st["U"] = _sequences(case, P, u0, st["instance"], seed).requires_grad_()
    return st


def run(state):
    s = state
    kind = s["kind"]
    if kind == "grad":
        S = aero.RolloutCost.apply(s["U"], s["planner"], s["instance"])
        (G,) = torch.autograd.grad(S.sum(), s["U"])
        return [S.detach(), G]
    s["u"].copy_(s["u0"])
    if kind == "batch":
        s["batch"].plan(s["items"])
        k = s["keep"]
        # the fleet's updated nominals whole; the best sequence, costs and index of 16 planners
        return [s["u"]] + [list(x[2:]) for x in k[:16]]
    if kind == "flight":
        f = s["frames"][s["at"]]  # the ring comes round to the slot that holds this frame
        s["at"] = (s["at"] + 1) % len(s["frames"])
        s["acc"].push(*f)
        if s["cloud"] is None:
            cloud, _ = s["acc"].view()
        else:
            cloud = s["cloud"][:s["acc"].gather(s["cloud"])]
        s["planner"].plan_step(s["x"], cloud, s["goal"], s["P"], s["u"], *s["outs"])
        aero.shift_nominal(s["u"], s["shift"], s["scratch"])
        return [s["u"], *s["outs"]]
    if s["entry"] == "noalloc":
        aero.plan_step_noalloc(s["x"], s["cloud"], s["goal"], s["P"], s["u"], *s["outs"])
    elif s["entry"] == "host":
        s["planner"].plan_step_host(s["x"], s["cloud"], s["goal"], s["P"], s["u"], *s["outs"])
    else:
        s["planner"].plan_step(s["x"], s["cloud"], s["goal"], s["P"], s["u"], *s["outs"])
    return [s["u"], *s["outs"]]


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [work(s) for s in _batch_items(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if kind == "grad":
        steps = case["seqs"] * case["T"]
        return {"bytes": 32.0 * steps + 4.0 * case["seqs"], "flops": FLOPS_GRAD * steps}
    s = _as_step(case) if kind == "flight" else case
    E, K, T = s["M_h"] * s["M_v"], s["K"], s["T"]
    b = 12.0 * s["n"] + 32.0 * E * T + 16.0 * T + 4.0 * E + 4
    if kind == "flight":
        b += 24.0 * case["n"] + 32.0 * E * T
    f = (FLOPS_STEP * K * s["iters"] + FLOPS_STAGE2 + FLOPS_GRAD * s["refine"]) * E * T + 20.0 * s["n"]
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits (plain torch and numpy)
# ---------------------------------------------------------------------------

def _rot32(q):
    """R(q) in binary32, nine products and the sums (the partition's decisions use it)."""
    w, x, y, z = (np.float32(a) for a in q)
    one, two = np.float32(1), np.float32(2)
    xx, yy, zz, xy, xz, yz, wx, wy, wz = x * x, y * y, z * z, x * y, x * z, y * z, w * x, w * y, w * z
    return np.array([[one - two * (yy + zz), two * (xy - wz), two * (xz + wy)],
                     [two * (xy + wz), one - two * (xx + zz), two * (yz - wx)],
                     [two * (xz - wy), two * (yz + wx), one - two * (xx + yy)]], np.float32)


def _body(R, d):
    """R^T d with every product and sum rounded to binary32."""
    c = [d[:, i] for i in range(3)]
    return [(float(R[0, i]) * c[0] + float(R[1, i]) * c[1]) + float(R[2, i]) * c[2] for i in range(3)]


def _bin(guess, lo, hi, s):
    """The largest bin of [lo, hi] whose edge predicate s(k) >= 0 holds, else lo, from a guess."""
    k = torch.minimum(torch.maximum(guess, lo), hi)
    for _ in range(2):
        up = (k < hi) & (s(torch.minimum(k + 1, hi)) >= 0)
        down = ~up & (k > lo) & (s(k) < 0)
        k = k + up.long() - down.long()
    return k


def _cones(R, d, A, El):
    """(fine cone, binary32 squared range) of displacements d (n x 3 float32)."""
    th = np.pi * (2 * np.arange(A) - A) / A
    lo, hi = (float(np.float32(x)) for x in (-math.pi / 2, math.pi / 2))
    ph = lo + ((hi - lo) * np.arange(El + 1)) / El
    ca, sa, ce, se = (torch.from_numpy(f(a)).float().to(DEV)
                      for a, f in ((th, np.cos), (th, np.sin), (ph, np.cos), (ph, np.sin)))
    bx, by, bz = _body(R, d)
    rxy2 = bx * bx + by * by
    r2 = rxy2 + bz * bz
    rho = rxy2.sqrt()
    upper = (by > 0) | ((by == 0) & (bx > 0))
    half = A // 2
    lo_k = torch.where(upper, half, 0)
    hi_k = torch.where(upper, A - 1, half - 1)
    az = torch.floor((torch.atan2(by.double(), bx.double()) + math.pi) * (A / (2 * math.pi))).long()
    ia = _bin(az, lo_k, hi_k, lambda k: by * ca[k] - bx * sa[k])
    el = torch.floor((torch.atan2(bz.double(), rho.double()) - lo) * (El / (hi - lo))).long()
    je = _bin(el, torch.zeros_like(el), torch.full_like(el, El - 1), lambda k: bz * ce[k] - rho * se[k])
    return je * A + ia, r2


def _context(P, cloud, p, q, v, goal):
    """Collision points (relative to p), guides and the start, in 64 bits."""
    A, El, Pa, Pe = P["fine_az"], P["fine_el"], P["pool_az"], P["pool_el"]
    R = _rot32(q)
    f = lambda x: float(np.float32(x))  # noqa: E731
    rmax2 = float(np.float32(P["r_max"]) * np.float32(P["r_max"]))
    idx = torch.isfinite(cloud).all(1).nonzero()[:, 0]
    d = cloud[idx] - torch.from_numpy(p).to(DEV)
    keep = torch.empty(len(d), dtype=torch.bool, device=DEV)
    cone = torch.empty(len(d), dtype=torch.long, device=DEV)
    key = torch.empty(len(d), dtype=torch.long, device=DEV)
    for s in range(0, len(d), 1 << 21):
        t = slice(s, s + (1 << 21))
        cone[t], r2 = _cones(R, d[t], A, El)
        keep[t] = (r2 > 0) & (r2 <= rmax2)
        key[t] = (r2.contiguous().view(torch.int32).long() << 32) | idx[t]
    empty = (1 << 63) - 1
    keys = torch.full((A * El,), empty, dtype=torch.long, device=DEV)
    keys.scatter_reduce_(0, cone[keep], key[keep], "amin")
    if P["collision_set"]:
        pts = d[keep].double()
    else:
        won = keys[keys < empty] & 0xFFFFFFFF
        pts = (cloud[won] - torch.from_numpy(p).to(DEV)).double()
    # coarse winners: larger range, then nearer the coarse centre, then lower index
    rk = torch.where(keys == empty, int(np.float32(rmax2).view(np.int32)), keys >> 32).cpu().numpy()
    rk = rk.reshape(El, A)
    Ac, Ec = A // Pa, El // Pe
    gd = torch.from_numpy((goal - p).astype(np.float32)[None]).to(DEV)
    gcell = int(_cones(R, gd, A, El)[0][0])
    Ig, Jg = (gcell % A) // Pa, (gcell // A) // Pe
    E, T = P["E"], P["T"]
    dt, ell = f(P["dt"]), f(P["ell"])
    Tg = T * dt
    v_end = f(P["v_end"]) if P["v_end"] > 0 else ell / Tg
    lo, hi = (f(x) for x in (-math.pi / 2, math.pi / 2))
    guides = np.zeros((E, T, 3))
    s = (np.arange(T) + 1) / T
    for e in range(E):
        m, n = e % P["M_h"], e // P["M_h"]
        I = (Ig + m - P["M_h"] // 2) % Ac
        J = min(max(Jg + n - P["M_v"] // 2, 0), Ec - 1)
        best = None
        for b in range(Pe):
            for a in range(Pa):
                j, i = J * Pe + b, I * Pa + a
                cand = (-int(rk[j, i]), abs(2 * a + 1 - Pa) + abs(2 * b + 1 - Pe), j * A + i)
                best = cand if best is None or cand < best else best
        j, i = best[2] // A, best[2] % A
        al, be = math.pi * (-1 + (2 * i + 1) / A), lo + (j + 0.5) * (hi - lo) / El
        w = np.array([math.cos(be) * math.cos(al), math.cos(be) * math.sin(al), math.sin(be)])
        pr = ell * (R.astype(np.float64) @ w)
        V0, V1 = v.astype(np.float64) * Tg, v_end / np.linalg.norm(pr) * pr * Tg
        for r in range(3):
            co = [6 * pr[r] - 3 * V0[r] - 3 * V1[r], -15 * pr[r] + 8 * V0[r] + 7 * V1[r],
                  10 * pr[r] - 6 * V0[r] - 4 * V1[r], 0.0, V0[r], 0.0]
            guides[e, :, r] = np.polyval(co, s)
    x0 = [torch.from_numpy(a.astype(np.float64)).to(DEV) for a in (np.zeros(3), q, v)]
    return dict(pts=pts, guides=torch.from_numpy(guides).to(DEV), x0=x0, dt=dt,
                goal=torch.from_numpy((goal - p).astype(np.float32).astype(np.float64)).to(DEV),
                P={k: ([f(a) for a in x] if isinstance(x, list) else f(x) if isinstance(x, float) else x)
                   for k, x in P.items()})


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 words of 64-bit tensors of 32-bit counters (broadcast)."""
    m32 = 0xFFFFFFFF
    c = list(torch.broadcast_tensors(c0, c1, torch.tensor(c2, device=DEV), torch.tensor(c3, device=DEV)))
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # the low 64 bits, wrapped
        c = [((b >> 32) & m32) ^ c[1] ^ k0, b & m32, ((a >> 32) & m32) ^ c[3] ^ k1, a & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _noise(P, e, it):
    """Perturbations K x T x 4 of instance e."""
    k = torch.arange(P["K"], device=DEV)[:, None]
    j = torch.arange(P["T"], device=DEV)[None]
    w = _philox(k, j, e, (P["step_id"] << 8) | it, P["seed"])
    u = [(2 * (x >> 9) + 1).double() * 2.0 ** -24 for x in w]
    out = []
    for a, b in ((0, 1), (2, 3)):
        r = torch.sqrt(-2 * torch.log(u[a]))
        out += [r * torch.cos(2 * math.pi * u[b]), r * torch.sin(2 * math.pi * u[b])]
    return torch.stack(out, -1) * torch.tensor(P["sigma"], dtype=torch.float64, device=DEV)


def _rates(q, u, g, mass):
    """Attitude and velocity rates of the quadrotor model."""
    w, x, y, z = q.unbind(-1)
    F, a, b, c = u.unbind(-1)
    dq = 0.5 * torch.stack([-x * a - y * b - z * c, w * a + y * c - z * b, w * b - x * c + z * a,
                            w * c + x * b - y * a], -1)
    f = F / mass
    dv = torch.stack([f * 2 * (x * z + w * y), f * 2 * (y * z - w * x), f * (1 - 2 * (x * x + y * y)) - g], -1)
    return dq, dv


def _rollout(C, U):
    """States after each step of U (B x T x 4): p, q, v as B x T x n."""
    P, h = C["P"], C["dt"]
    p, q, v = (x.expand(len(U), -1) for x in C["x0"])
    out = []
    for t in range(U.shape[1]):
        u = U[:, t]
        kq, kv, kp = [], [], []
        for w in (0.0, 0.5, 0.5, 1.0):
            qs = q + w * h * kq[-1] if kq else q
            kp.append(v + w * h * kv[-1] if kv else v)
            dq, dv = _rates(qs, u, P["g"], P["mass"])
            kq.append(dq)
            kv.append(dv)
        rk = lambda k: h / 6 * (k[0] + 2 * k[1] + 2 * k[2] + k[3])  # noqa: E731
        p, q, v = p + rk(kp), q + rk(kq), v + rk(kv)
        q = q / (q * q).sum(-1, keepdim=True).sqrt()
        out.append((p, q, v))
    return [torch.stack([o[i] for o in out], 1) for i in range(3)]


def _nearest(C, p):
    """Index of the nearest collision point of every query (N x 3)."""
    pts = C["pts"]
    idx = torch.empty(len(p), dtype=torch.long, device=DEV)
    n = max(1, (1 << 27) // max(1, len(pts)))
    for s in range(0, len(p), n):
        a = p[s:s + n]
        d = a[:, :1] - pts[:, 0]
        d *= d
        for i in (1, 2):
            e = a[:, i:i + 1] - pts[:, i]
            d.addcmul_(e, e)
        idx[s:s + n] = d.argmin(1)
    return idx


def _norm(x):
    """|x| over the last axis with a zero gradient at zero."""
    n = (x * x).sum(-1)
    ok = n > 0
    return torch.where(ok, torch.where(ok, n, torch.ones_like(n)).sqrt(), torch.zeros_like(n))


def _cost(C, X, U=None, guide=None):
    """Sum over the horizon of the state terms (Stage II), with U and guide of S(1)."""
    P = C["P"]
    p, q, v = X
    vg, qg = (torch.tensor(P[k], dtype=torch.float64, device=DEV) for k in ("v_goal", "q_goal"))
    w, x, y, z = q.unbind(-1)
    r = torch.stack([-w * qg[1] + x * qg[0] - y * qg[3] + z * qg[2],
                     -w * qg[2] + x * qg[3] + y * qg[0] - z * qg[1],
                     -w * qg[3] - x * qg[2] + y * qg[1] + z * qg[0]], -1)
    c = P["Q_p"] * _norm(p - C["goal"]) + P["Q_v"] * _norm(v - vg) + P["Q_q"] * 8 ** 0.5 * _norm(r)
    if len(C["pts"]):
        near = C["pts"][_nearest(C, p.detach().reshape(-1, 3))].reshape(p.shape)
        d = _norm(p - near)
        jc = torch.where(d < P["d_min"], torch.full_like(d, P["C_col"]),
                         P["C_col"] * torch.exp(-P["a_col"] * (d - P["d_min"])))
        c = c + torch.where(d < P["d_max"], jc, torch.zeros_like(d))
    S = c.sum(1)
    if U is None:
        return S
    S = S + (P["Q_track"] * _norm(p - guide) + P["Q_vnorm"] * (v * v).sum(-1)).sum(1)
    S = S + P["Q_c"] * (U[:, :-1] ** 2).sum((1, 2))
    return S + P["Q_cd"] * ((U[:, 1:-1] - U[:, :-2]) ** 2).sum((1, 2))


def _cost_grad(C, U, e):
    U = U.detach().requires_grad_()
    S = _cost(C, _rollout(C, U), U, C["guides"][e])
    (G,) = torch.autograd.grad(S.sum(), U)
    return S.detach(), G


def _plan(P32, cloud, p, q, v, goal, u0):
    C = _context(P32, cloud, p, q, v, goal)
    P = C["P"]
    E, K, T = P["E"], P["K"], P["T"]
    lo, hi = (torch.tensor(P[k], dtype=torch.float64, device=DEV) for k in ("u_min", "u_max"))
    u = u0.to(DEV).double()
    with torch.no_grad():
        for it in range(P["iters"]):
            U = torch.empty((E, K, T, 4), dtype=torch.float64, device=DEV)
            S = torch.empty((E, K), dtype=torch.float64, device=DEV)
            for e in range(E):
                U[e] = torch.minimum(torch.maximum(u[e] + _noise(P, e, it), lo), hi)
            per = max(1, (1 << 21) // (K * T))  # instances rolled out together
            for e in range(0, E, per):
                Ue = U[e:e + per].reshape(-1, T, 4)
                g = C["guides"][e:e + per, None].expand(-1, K, -1, -1).reshape(-1, T, 3)
                S[e:e + per] = _cost(C, _rollout(C, Ue), Ue, g).reshape(-1, K)
            w = torch.softmax(-(S - S.amin(1, keepdim=True)) / P["lam"], 1)
            u = u + torch.einsum("ek,ektc->etc", w, U - u[:, None])
    for _ in range(P["refine_steps"]):
        for e in range(E):
            _, G = _cost_grad(C, u[e:e + 1], e)
            u[e] = torch.minimum(torch.maximum(u[e] - P["refine_step"] * G[0], lo), hi)
    with torch.no_grad():
        S2 = _cost(C, _rollout(C, u))
    return C, u, S2


def _too_long(c):
    """Whether the brute-force nearest points would take over about 20 seconds."""
    s = c if c["kind"] == "step" else _as_step(c)
    A = PARTITIONS[s["part"]]
    pts = s["n"] if s["raw"] else min(s["n"], A["fine_az"] * A["fine_el"])
    q = s["M_h"] * s["M_v"] * s["K"] * s["T"] * s["iters"]
    return q * pts > 4e11


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        steps = _batch_items(case)
        if sum(s["M_h"] * s["M_v"] * s["K"] * s["T"] * 4000 for s in steps) > 4e11:
            return None
        us, rest = [], []
        for i, s in enumerate(steps):
            _, u, S2 = _plan(*_step_inputs(s, seed * 64 + i))
            us.append(u.reshape(-1))
            rest.append([u[int(S2.argmin())], S2, None])
        return [torch.cat(us)] + rest[:16]
    if _too_long(case):
        return None
    if kind == "grad":
        s = _as_step(case)
        P, cloud, p, q, v, goal, u0 = _step_inputs(s, seed)
        C = _context(P, cloud, p, q, v, goal)
        e = P["E"] // 2
        S, G = _cost_grad(C, _sequences(case, P, u0, e, seed).double(), e)
        return [S, G]
    if kind == "flight":
        P, frames, p, q, v, goal, u0 = _flight_inputs(case, seed)
        parts = []
        for pts, fp, fq in frames:
            qd = fq.astype(np.float64) / np.linalg.norm(fq.astype(np.float64))
            R = _rot32(qd.astype(np.float32))
            rows = [float(fp[i]) + ((float(R[i, 0]) * pts[:, 0] + float(R[i, 1]) * pts[:, 1])
                                    + float(R[i, 2]) * pts[:, 2]) for i in range(3)]
            parts.append(torch.stack(rows, 1))
        _, u, S2 = _plan(P, torch.cat(parts), p, q, v, goal, u0)
        m = max(1, round(0.1 / case["dt"]))
        at = torch.clamp(torch.arange(P["T"], device=DEV) + m, max=P["T"] - 1)
        return [u[:, at], u[int(S2.argmin())], S2, None]
    _, u, S2 = _plan(*_step_inputs(case, seed))
    return [u, u[int(S2.argmin())], S2, None]
