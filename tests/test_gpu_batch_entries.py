"""A batched call's candidate entries are the points themselves or, where the lists are
pruned (enough sample-steps and no every-point set in the call), item indices: in
both forms, both Stage I passes and the refinement, every Stage II cost is the oracle's
over the planner's collision set and the lists hold the set's points."""
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


@pytest.mark.parametrize("lanes", [1, 4])
@pytest.mark.parametrize("K,raw,refine", [(256, (0, 0, 0), 1), (256, (1, 0, 1), 1), (2048, (0, 0, 0), 1),
                                          (2048, (0, 1, 0), 0), (2048, (0, 0, 0), 0)])
def test_stage2_over_each_set(aero, orc, K, raw, refine, lanes):
    import torch
    dev = torch.device("cuda")
    ws = []
    for i, r in enumerate(raw):
        w = I.make_workload("ensemble", seed=i)
        rng = np.random.default_rng([K, i])
        n = 500 + 700 * i      # a wall beside the flight line
        wall = np.stack([rng.uniform(0.5, 4.0, n), np.full(n, 0.7) + rng.uniform(-0.05, 0.05, n),
                         rng.uniform(0.5, 2.5, n)], 1)
        w.cloud = np.concatenate([w.cloud[::3], wall]).astype(np.float32)
        w.params.update(E=8, M_h=4, M_v=2, K=K, T=40, collision_set=r, lanes_per_sample=lanes, refine_steps=refine,
                        refine_step=1e-3, step_id=i)
        ws.append(w)
    P = ws[0].params
    b = aero.Batch(len(ws), E_max=8, K_max=K, T_max=40, fine_cells_max=P["fine_az"] * P["fine_el"],
                   n_points_max=max(len(w.cloud) for w in ws))
    keep, items = [], []
    for w in ws:
        k = (torch.from_numpy(w.cloud).to(dev), torch.from_numpy(w.hover_nominal()).to(dev),
             torch.empty((40, 4), device=dev), torch.empty((8,), device=dev),
             torch.empty((1,), dtype=torch.int32, device=dev))
        keep.append(k)
        items.append(aero.Batch.item(aero.state_struct(w.p0, w.q0, w.v0), k[0], w.goal, aero.params_struct(w.params),
                                     *k[1:]))
    b.plan(items)
    torch.cuda.synchronize()
    assert b.sync_status() == 0
    entries = [b.debug(i, "GRID_POINTS") for i in range(len(ws))]
    b.close()
    near = compared = 0
    for w, k, ent in zip(ws, keep, entries):
        keys = orc.partition(w.cloud, w.p0, w.q0, w.params)[0]
        pts = orc.collision_set(w.cloud, w.p0, w.q0, keys, w.params)
        rel = {tuple(p) for p in (w.cloud - w.p0).astype(np.float32)}
        assert len(ent) > 0 and all(tuple(e[:3]) in rel for e in ent[::97])
        U, c = k[1].cpu().numpy().astype(np.float64), k[3].cpu().numpy()
        for e in range(8):
            X = orc.rollout(x0_of(w), U[e], P["dt"], P["mass"], P["g"])
            t = orc.cost_terms(X, U[e], None, w.goal.astype(np.float64), pts, w.params, stage=2, want_dist=True)
            d = t["dist"]
            if min(np.abs(d - P["d_min"]).min(), np.abs(d - P["d_max"]).min()) <= JUMP_BAND:
                continue
            assert abs(c[e] - t["S"]) <= TOL_COST_REL * abs(t["S"]), e
            compared += 1
            near += t["J_col"] > 0
        assert int(k[4][0]) == int(np.argmin(c))
    assert compared >= 12 and near >= 4
