"""The collision grid's lists are pruned to the entries that can be a query's
nearest: every sampled state's nearest-point distance is still the minimum over
the whole collision set, for lists around the sizes at which the pruning
changes its form (whole below 5, groups of lanes up to 8 and 16, the seeds from the
first 128, more than 640 kept), with duplicated and equidistant points, on
fine and coarse cells and in both Stage I passes."""
import numpy as np
import pytest

from paper_2509_17340_gb300 import inputs as I
from gpu_util import run_gpu

pytestmark = pytest.mark.gpu

# The kernel's squared distance differs from the exact one of the same binary32
# states and points by the rounding of three differences, products and sums:
# below 4 * 2^-24 relative, half of that for the distance.
TOL_REL = 2.4e-7


@pytest.fixture(scope="module")
def aero():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_17340_gb300 import build
    build.build()
    from paper_2509_17340_gb300 import aero as A
    return A


def _cloud(kind, n, p0, rng):
    if kind == "sheet":        # a wall ahead: most entries lie behind nearer ones
        p = np.stack([np.full(n, 1.6), rng.uniform(-0.8, 0.8, n), rng.uniform(-0.8, 0.8, n)], 1)
    elif kind == "cluster":    # within half a cell, every third point a duplicate
        p = np.array([1.2, 0.3, 0.2]) + rng.uniform(-0.2, 0.2, (n, 3))
        p[::3] = p[1 % n]
    else:                      # a lattice: exactly equidistant neighbours
        p = np.round(np.array([1.3, 0.0, 0.0]) + rng.uniform(-0.7, 0.7, (n, 3)), 1)
    p[0] = [1.4, 0.2, 0.1]     # beside the flight line
    return (p0 + p).astype(np.float32)


@pytest.mark.parametrize("lanes", [1, 4])
@pytest.mark.parametrize("r_max", [10.0, 60.0])
@pytest.mark.parametrize("kind", ["sheet", "cluster", "lattice"])
@pytest.mark.parametrize("n", [1, 4, 5, 8, 9, 16, 17, 128, 129, 640, 641, 3000])
def test_nearest_distance_is_the_minimum_over_the_set(aero, n, kind, r_max, lanes):
    w = I.make_workload("plain", seed=n)
    rng = np.random.default_rng([n, lanes])
    w.cloud = _cloud(kind, n, w.p0, rng)
    w.v0 = np.array([2.0, 0.0, 0.0], np.float32)
    P = w.params
    P.update(E=1, M_h=1, M_v=1, K=2304, T=20, r_max=r_max, collision_set=1, lanes_per_sample=lanes,
             debug_samples=64, sigma=[2.0, 1.5, 1.5, 1.5])
    pl = aero.Planner(E_max=1, K_max=2304, T_max=20, fine_cells_max=P["fine_az"] * P["fine_el"],
                      n_points_max=n, debug_samples_max=64)
    try:
        run_gpu(aero, pl, w, P, w.hover_nominal())
        x = pl.debug("SAMPLE_X").reshape(64, 21, 10)[:, 1:, :3].astype(np.float64)
        got = pl.debug("SAMPLE_DIST").reshape(64, 20).astype(np.float64)
    finally:
        pl.close()
    rel = (w.cloud - w.p0).astype(np.float32).astype(np.float64)
    want = np.sqrt(((x[:, :, None] - rel) ** 2).sum(-1)).min(-1)
    near = want < P["d_max"]
    edge = np.abs(want - P["d_max"]) < 1e-6
    assert np.array_equal((got < np.inf)[~edge], near[~edge])
    both = near & (got < np.inf)
    assert both.sum() > 0
    assert (np.abs(got - want)[both] <= TOL_REL * want[both]).all()
