"""The partition at the ends of what its parameters accept: a range bound whose square is
infinite in binary32, where finite points beyond 1.8e19 m are inside and non-finite ones
are still left out; elevation spans of more than a turn, whose cones are wider than half
a turn."""
import numpy as np
import pytest

from paper_2509_17340_gb300 import inputs as I
from gpu_util import run_gpu
from test_gpu_partition_edges import aero  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


def _step(aero, w, P):  # noqa: F811
    pl = aero.Planner(E_max=1, K_max=32, T_max=4, fine_cells_max=P["fine_az"] * P["fine_el"],
                      n_points_max=len(w.cloud), debug_samples_max=1)
    try:
        return run_gpu(aero, pl, w, P, w.hover_nominal())
    finally:
        pl.close()


@pytest.mark.parametrize("turned", [False, True])
@pytest.mark.parametrize("A,El", [(6, 3), (120, 60)])
@pytest.mark.parametrize("r_max", [1e10, 1e19, 1e20])
def test_range_bound_beyond_binary32(aero, orc, r_max, A, El, turned):  # noqa: F811
    w = I.make_workload("plain", seed=A)
    rng = np.random.default_rng([A, turned])
    w.p0 = np.zeros(3, np.float32)
    if turned:
        w.q0 = I.random_unit_quaternion(rng)
    n = 6000
    d = rng.normal(size=(n, 3))
    p = d / np.linalg.norm(d, axis=1, keepdims=True) * 10.0 ** rng.uniform(-2, 20, (n, 1))
    p[:600] *= 10.0 ** rng.uniform(0, 18, (600, 1))       # up to 10^38
    p = p.astype(np.float32)
    bad = rng.permutation(n)[:300]
    p[bad, rng.integers(0, 3, 300)] = np.array([np.inf, -np.inf, np.nan], np.float32)[np.arange(300) % 3]
    w.cloud = p
    P = w.params
    P.update(E=1, M_h=1, M_v=1, K=32, T=4, fine_az=A, fine_el=El, pool_az=1, pool_el=1, r_max=r_max)
    keys, kept = orc.partition(w.cloud, w.p0, w.q0, P)
    g = _step(aero, w, P)
    assert list(g["point_counts"]) == [n, 300, kept]
    assert np.array_equal(g["keys"], keys)


@pytest.mark.parametrize("El,lo,hi", [(2, -6.0, 2.0), (2, -2.0, 6.0), (3, -5.0, 5.0), (1, -10.0, 10.0), (3, -4.0, 4.0)])
def test_cones_wider_than_half_a_turn(aero, orc, El, lo, hi):  # noqa: F811
    w = I.make_workload("plain", seed=El)
    rng = np.random.default_rng([El, int(10 * hi)])
    w.p0 = np.zeros(3, np.float32)
    d = rng.normal(size=(6000, 3))
    w.cloud = (d / np.linalg.norm(d, axis=1, keepdims=True) * rng.uniform(0.1, 9.0, (6000, 1))).astype(np.float32)
    P = w.params
    P.update(E=1, M_h=1, M_v=1, K=32, T=4, fine_az=120, fine_el=El, pool_az=1, pool_el=1, el_lo=lo, el_hi=hi)
    keys, kept = orc.partition(w.cloud, w.p0, w.q0, P)
    g = _step(aero, w, P)
    assert list(g["point_counts"]) == [6000, 0, kept]
    assert np.array_equal(g["keys"], keys)
