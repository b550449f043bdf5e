"""Lists of a single planner's step are pruned where the samples meet long ones (the list
probe): the same wall beside the flight line and out of reach, both collision sets and
both Stage I passes.  The pruned lists hold the kept entries last, and on either side of
the decision every sampled state's distance is the minimum over the whole set."""
import numpy as np
import pytest

from paper_2509_17340_gb300 import inputs as I
from gpu_util import run_gpu
from test_gpu_pruned_lists import TOL_REL, _cloud, aero  # noqa: F401  (aero: the fixture)

pytestmark = pytest.mark.gpu


def _kept_last(pl):
    """Of the lists of 20 entries and more, the share whose entry nearest to the cell's
    centre (a seed, so kept) is in the second half."""
    start = pl.debug("GRID_START")
    pts = pl.debug("GRID_POINTS").reshape(-1, 4)[:, :3]
    meta = pl.debug("GRID_META")
    G, (origin, h) = int(meta[0]), meta[4:6].view(np.float32)
    n = np.diff(start)
    late = []
    for c in np.flatnonzero((n >= 20) & (n <= 128)):
        m = origin + (np.array([c % G, c // G % G, c // (G * G)]) + 0.5) * h
        d = ((pts[start[c]:start[c + 1]] - m) ** 2).sum(1)
        late.append(np.argmin(d) >= n[c] // 2)
    return float(np.mean(late)), len(late)


@pytest.mark.parametrize("near", [True, False])
@pytest.mark.parametrize("lanes", [1, 4])
@pytest.mark.parametrize("raw", [0, 1])
def test_both_sides_of_the_probe(aero, raw, lanes, near):  # noqa: F811
    w = I.make_workload("ensemble", seed=3)
    P = w.params
    n = 4_000 if raw else 130_000
    P.update(E=8, M_h=4, M_v=2, K=1024, T=40, fine_az=120, fine_el=60, pool_az=6, pool_el=6, collision_set=raw,
             lanes_per_sample=lanes, debug_samples=32)
    rng = np.random.default_rng([raw, lanes])
    w.p0, w.v0 = np.zeros(3, np.float32), np.array([1.0, 0.0, 0.0], np.float32)
    side = 0.9 if near else -8.0
    w.cloud = np.stack([rng.uniform(-0.5, 2.5, n), side + rng.uniform(-0.1, 0.1, n), rng.uniform(-2, 1, n)],
                       1).astype(np.float32)
    pl = aero.Planner(E_max=8, K_max=1024, T_max=40, fine_cells_max=120 * 60, n_points_max=n, debug_samples_max=32)
    try:
        pl.profile(True)
        g = run_gpu(aero, pl, w, P, w.hover_nominal())
        launches = pl.profile_read()["grid"][1]
        late, lists = _kept_last(pl)
    finally:
        pl.close()
    assert launches == 4 and lists >= 20
    assert late > 0.95 if near else late < 0.8
    if raw:
        pts = w.cloud.astype(np.float64)
    else:
        keys = g["keys"][g["keys"] != np.uint64(0xFFFFFFFFFFFFFFFF)]
        pts = w.cloud[(keys & np.uint64(0xFFFFFFFF)).astype(np.int64)].astype(np.float64)
    x, got = g["sX"][:, :, 1:, :3].reshape(-1, 3), g["sD"].reshape(-1)
    hit = 0
    for s in range(0, len(x), 512):
        want = np.sqrt(((x[s:s + 512, None] - pts) ** 2).sum(-1).min(-1))
        d, inside = got[s:s + 512], want < P["d_max"]
        edge = np.abs(want - P["d_max"]) < 1e-6
        assert np.array_equal((d < np.inf)[~edge], inside[~edge])
        both = inside & (d < np.inf)
        assert (np.abs(d - want)[both] <= TOL_REL * want[both]).all()
        hit += both.sum()
    assert hit > 0 if near else True


@pytest.mark.parametrize("n", [4, 5, 8, 9, 16, 17, 128, 129, 640, 641, 3000])
@pytest.mark.parametrize("kind", ["sheet", "cluster", "lattice"])
def test_pruned_lists_of_every_length(aero, n, kind):  # noqa: F811
    """Lists around the sizes at which the pruning changes its form (whole below 5, groups
    of lanes up to 8 and 16, the seeds from the first 128, more than 640 kept), met often
    enough to be pruned."""
    w = I.make_workload("plain", seed=n)
    rng = np.random.default_rng([n, 7])
    w.cloud = _cloud(kind, n, w.p0, rng)
    w.v0 = np.array([2.0, 0.0, 0.0], np.float32)
    P, K, lanes = w.params, 1 << 16, 1 if n % 2 else 4
    P.update(E=1, M_h=1, M_v=1, K=K, T=20, collision_set=1, lanes_per_sample=lanes, debug_samples=64,
             sigma=[2.0, 1.5, 1.5, 1.5])
    pl = aero.Planner(E_max=1, K_max=K, T_max=20, fine_cells_max=P["fine_az"] * P["fine_el"], n_points_max=n,
                      debug_samples_max=64)
    try:
        g = run_gpu(aero, pl, w, P, w.hover_nominal())
        if n >= 640:
            late, lists = _kept_last(pl)
            assert lists == 0 or late > 0.95
    finally:
        pl.close()
    x, got = g["sX"][0, :, 1:, :3] - w.p0.astype(np.float64), g["sD"][0]
    rel = (w.cloud - w.p0).astype(np.float32).astype(np.float64)
    want = np.sqrt(((x[:, :, None] - rel) ** 2).sum(-1)).min(-1)
    near, edge = want < P["d_max"], np.abs(want - P["d_max"]) < 1e-6
    assert np.array_equal((got < np.inf)[~edge], near[~edge])
    both = near & (got < np.inf)
    assert both.sum() > 0
    # (the states are stored relative to the start; adding and taking it off again rounds)
    assert (np.abs(got - want)[both] <= TOL_REL * want[both] + 1e-9).all()
