"""A one-lane step whose Stage I CTAs all fit on the GPU at once: the update launch's
CTAs start while the grid is still being written (and its lists pruned), and their
warm-up runs must not touch it.  Steps on alternating clouds follow one another without
a wait; every Stage II cost is the oracle's over the whole collision set."""
import numpy as np
import pytest

from paper_2509_17340_gb300 import inputs as I
from gpu_util import JUMP_BAND, TOL_COST_REL, x0_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def aero():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_17340_gb300 import build
    build.build()
    from paper_2509_17340_gb300 import aero as A
    return A


def _cloud(w, side, rng):
    """The forest sweep and, beside the flight line on one side, 4,000 points of a wall."""
    n = 4000
    wall = np.stack([rng.uniform(0.5, 4.0, n), np.full(n, side) + rng.uniform(-0.05, 0.05, n),
                     rng.uniform(0.5, 2.5, n)], 1)
    return np.concatenate([w.cloud * np.array([1.0, np.sign(side), 1.0]), wall]).astype(np.float32)


@pytest.mark.parametrize("refine", [0, 2])
def test_stage2_over_the_whole_set(aero, orc, refine):
    import torch
    w = I.make_workload("ensemble")
    P = w.params
    P.update(E=8, M_h=4, M_v=2, K=8192, T=20, collision_set=1, lanes_per_sample=1, refine_steps=refine,
             refine_step=1e-3)
    rng = np.random.default_rng(3)
    clouds = [_cloud(w, s, rng) for s in (0.7, -0.75)]
    assert P["E"] * P["K"] * P["T"] >= 14 * len(clouds[0])        # such a set is pruned
    pl = aero.Planner(E_max=8, K_max=8192, T_max=20, fine_cells_max=P["fine_az"] * P["fine_el"],
                      n_points_max=len(clouds[0]))
    dev = torch.device("cuda")
    xs = [torch.from_numpy(c).to(dev) for c in clouds]
    u0 = torch.from_numpy(np.ascontiguousarray(w.hover_nominal()[:, :20])).to(dev)
    runs, state = [], aero.state_struct(w.p0, w.q0, w.v0)
    for s in range(12):
        out = (u0.clone(), torch.empty((20, 4), device=dev), torch.empty((8,), device=dev),
               torch.empty((1,), dtype=torch.int32, device=dev))
        runs.append(out)
    torch.cuda.synchronize()
    for s, out in enumerate(runs):
        pl.plan_step(state, xs[s & 1], w.goal, aero.params_struct(dict(P, step_id=s)), *out)
    torch.cuda.synchronize()
    assert pl.sync_status() == 0
    pl.close()
    sets = [orc.collision_set(c, w.p0, w.q0, orc.partition(c, w.p0, w.q0, P)[0], P) for c in clouds]
    near = compared = 0
    for s, (un, _, cand, best) in enumerate(runs):
        U, c = un.cpu().numpy().astype(np.float64), cand.cpu().numpy()
        for e in range(8):
            X = orc.rollout(x0_of(w), U[e], P["dt"], P["mass"], P["g"])
            t = orc.cost_terms(X, U[e], None, w.goal.astype(np.float64), sets[s & 1], P, stage=2, want_dist=True)
            d = t["dist"]
            if min(np.abs(d - P["d_min"]).min(), np.abs(d - P["d_max"]).min()) <= JUMP_BAND:
                continue
            assert abs(c[e] - t["S"]) <= TOL_COST_REL * abs(t["S"]), (s, e)
            compared += 1
            near += t["J_col"] > 0
        assert int(best[0]) == int(np.argmin(c))
    assert compared >= 48 and near >= 12
