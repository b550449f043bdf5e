"""Pruned lists whose seeds are not unique: a lattice that is the same under exchange
of the axes, flown along its diagonal, where a cell's corners and centre have several
nearest entries at the same squared distance.  The seed must be one of them whole;
every sampled state's nearest-point distance is then the minimum over the set."""
import numpy as np
import pytest

from paper_2509_17340_gb300 import inputs as I
from gpu_util import run_gpu
from test_gpu_pruned_lists import TOL_REL, aero  # noqa: F401  (aero: the fixture)

pytestmark = pytest.mark.gpu


def _lattice(pitch):
    """Lattice points of the cube [0.3, 1.5]^3 with every exchange of their coordinates."""
    a = np.arange(0.3, 1.5, pitch)
    return np.stack(np.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3)


@pytest.mark.parametrize("pitch", [0.11, 0.15, 0.2])
def test_tied_seeds(aero, pitch):  # noqa: F811
    w = I.make_workload("plain", seed=1)
    rng = np.random.default_rng(0)
    p = _lattice(pitch).astype(np.float32)
    w.p0 = np.zeros(3, np.float32)      # the points' coordinates as they are
    w.cloud = p[rng.permutation(len(p))]
    w.v0 = np.array([1.6, 1.6, 1.6], np.float32)
    P = w.params
    K, D = 1 << 14, 1024      # sample-steps that meet enough entries for such a set to be pruned
    P.update(E=1, M_h=1, M_v=1, K=K, T=20, r_max=10.0, collision_set=1, lanes_per_sample=4,
             debug_samples=D, sigma=[2.0, 1.5, 1.5, 1.5])
    pl = aero.Planner(E_max=1, K_max=K, T_max=20, fine_cells_max=P["fine_az"] * P["fine_el"],
                      n_points_max=len(p), debug_samples_max=D)
    try:
        run_gpu(aero, pl, w, P, w.hover_nominal())
        x = pl.debug("SAMPLE_X").reshape(D, 21, 10)[:, 1:, :3].astype(np.float64)
        got = pl.debug("SAMPLE_DIST").reshape(D, 20).astype(np.float64)
    finally:
        pl.close()
    for s in range(0, D, 64):
        want = np.sqrt(((x[s:s + 64, :, None] - p.astype(np.float64)) ** 2).sum(-1)).min(-1)
        g, near = got[s:s + 64], want < P["d_max"]
        edge = np.abs(want - P["d_max"]) < 1e-6
        assert np.array_equal((g < np.inf)[~edge], near[~edge])
        both = near & (g < np.inf)
        assert (np.abs(g - want)[both] <= TOL_REL * want[both]).all()
