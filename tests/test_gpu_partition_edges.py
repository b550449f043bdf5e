"""The partition decides a point's cone from angle estimates when they are clear of
every edge, else from the exact predicates: points at all distances from the edges
(1e-2 to 1e-9 rad and on them), around the poles and the half planes, in geometries
from two cones to the finest, with full and partial elevation spans, get the
oracle's cones bit for bit."""
import numpy as np
import pytest

from paper_2509_17340_gb300 import inputs as I
from gpu_util import run_gpu

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


def _points(A, El, lo, hi, n, rng):
    """Body-frame points near the edges of the cones, at ranges of 0.01 to 9 m."""
    az = np.pi * (2 * rng.integers(0, A, n) - A) / A
    el = lo + (hi - lo) * rng.integers(0, El + 1, n) / El
    off = lambda: rng.choice([-1.0, 0.0, 1.0], n) * 10.0 ** rng.uniform(-9, -2, n)  # noqa: E731
    free = rng.integers(0, 3, n)      # 0: near an azimuth edge, 1: an elevation edge, 2: both
    az = np.where(free == 1, rng.uniform(-np.pi, np.pi, n), az + off())
    el = np.where(free == 0, rng.uniform(lo, hi, n), el + off())
    r = np.exp(rng.uniform(np.log(0.01), np.log(9.0), n))
    d = np.stack([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)], 1)
    # the poles and the half planes: tiny and zero lateral components
    m = n // 8
    d[:m, :2] *= 10.0 ** rng.uniform(-25, -3, (m, 1))
    d[m:m + 40, 0] = 0.0
    d[m + 40:m + 80, 1] = 0.0
    d[m + 80:m + 100, :2] = 0.0
    return r[:, None] * d


@pytest.mark.parametrize("turned", [False, True])
@pytest.mark.parametrize("A,El,lo,hi", [(2, 1, -np.pi / 2, np.pi / 2), (120, 60, -np.pi / 2, np.pi / 2),
                                        (512, 256, -np.pi / 2, np.pi / 2), (256, 64, -0.45, 0.6),
                                        (128, 64, 0.1, 0.101)])
def test_cones_near_edges(aero, orc, A, El, lo, hi, turned):
    w = I.make_workload("plain", seed=A + El)
    rng = np.random.default_rng([A, El, turned])
    lo, hi = float(np.float32(lo)), float(np.float32(hi))
    w.p0 = np.zeros(3, np.float32)
    if turned:
        w.q0 = I.random_unit_quaternion(rng)
    q = w.q0.astype(np.float64)
    x, y, z = q[1:]
    K = np.array([[0, -z, y], [z, 0, -x], [-y, x, 0]])
    R = np.eye(3) + 2 * q[0] * K + 2 * K @ K
    w.cloud = (_points(A, El, lo, hi, 60_000, rng) @ R.T).astype(np.float32)
    P = w.params
    P.update(E=1, M_h=1, M_v=1, K=32, T=4, fine_az=A, fine_el=El, pool_az=1, pool_el=1, el_lo=lo, el_hi=hi)
    pl = aero.Planner(E_max=1, K_max=32, T_max=4, fine_cells_max=A * El, n_points_max=len(w.cloud),
                      debug_samples_max=1)
    try:
        g = run_gpu(aero, pl, w, P, w.hover_nominal())
    finally:
        pl.close()
    keys, kept = orc.partition(w.cloud, w.p0, w.q0, P)
    assert np.array_equal(g["keys"], keys)
    assert list(g["point_counts"]) == [len(w.cloud), 0, kept]
