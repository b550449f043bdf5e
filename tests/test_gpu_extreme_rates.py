"""Noise-free rollouts at body rates where RK4 is unstable (dt |w| of about 7 and more):
the step's factor of the attitude is far from unit length, and a product of a
horizon's factors leaves binary32 unless they are normalised, while the attitude
itself, renormalised at every step, stays defined.  The cost-and-gradient entry
point takes any controls, Stage II the nominal within its bounds; both follow the oracle."""
import numpy as np
import pytest

from gpu_util import TOL_COST_REL, x0_of
from test_gpu_adjoint import TOL_GRAD, _case, _clear, _oracle_pts, aero  # noqa: F401  (aero: the fixture)

pytestmark = pytest.mark.gpu


def _sequences(P, rate, n, rng):
    """Hover with rates of this size about changing axes."""
    T = P["T"]
    u = np.zeros((n, T, 4), np.float32)
    u[..., 0] = P["mass"] * P["g"]
    axis = rng.normal(size=(n, 1, 3)) + 0.1 * rng.normal(size=(n, T, 3))
    u[..., 1:] = rate * axis / np.linalg.norm(axis, axis=-1, keepdims=True)
    u[0, : T // 2, 1:] *= 0.01      # flight-like, then a burst
    return u


@pytest.mark.parametrize("T", [33, 70, 128])
@pytest.mark.parametrize("rate", [60.0, 130.0, 150.0, 250.0, 400.0])
def test_cost_gradient_and_stage2(aero, orc, rate, T):  # noqa: F811
    import torch
    bound = [1000.0] * 3
    w = _case("refined", K=64, T=T, dt=0.05, refine_steps=0, sigma=[0.0] * 4, u_min=[0.0] + [-b for b in bound],
              u_max=[20.0] + bound)
    w.cloud = (w.p0 + np.array([[0.0, 0.0, 9.0]])).astype(np.float32)
    P = w.params
    rng = np.random.default_rng([int(rate), T])
    U = _sequences(P, rate, P["E"], rng)
    pl = aero.Planner(E_max=P["E"], K_max=64, T_max=T, fine_cells_max=P["fine_az"] * P["fine_el"], n_points_max=1)
    try:
        un = torch.from_numpy(U).cuda()
        ub, cand, best = aero.plan_step(pl, w.p0, w.q0, w.v0, torch.from_numpy(w.cloud).cuda(), w.goal, P, un)
        torch.cuda.synchronize()
        assert pl.sync_status() == 0
        guides = pl.debug("GUIDES").reshape(P["E"], T, 3).astype(np.float64) + w.p0
        assert np.array_equal(un.cpu().numpy(), U)      # no noise: the nominal is what it was
        S, G = torch.empty(P["E"], device="cuda"), torch.empty_like(un)
        pl.cost_grad(0, un, S, G)
        torch.cuda.synchronize()
    finally:
        pl.close()
    pts = _oracle_pts(orc, w)
    S, G, cand = S.cpu().numpy(), G.cpu().numpy().astype(np.float64), cand.cpu().numpy()
    checked = 0
    for e in range(P["E"]):
        u = U[e].astype(np.float64)
        ok, t = _clear(orc, w, u, guides[0], pts)
        if not ok:
            continue
        S_o, G_o = orc.cost_grad(x0_of(w), u, guides[0], w.goal.astype(np.float64), pts, P)
        assert abs(S[e] - S_o) <= TOL_COST_REL * abs(S_o), (e, S[e], S_o)
        assert np.abs(G[e] - G_o).max() <= TOL_GRAD * np.abs(G_o).max(), e
        X = orc.rollout(x0_of(w), u, P["dt"], P["mass"], P["g"])
        s2 = orc.cost_terms(X, u, None, w.goal.astype(np.float64), pts, P, stage=2)["S"]
        assert abs(cand[e] - s2) <= TOL_COST_REL * abs(s2), (e, cand[e], s2)
        checked += 1
    assert checked >= P["E"] // 2
