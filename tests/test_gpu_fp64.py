"""The FP64 path at the edges of its kernels: orders from 1 to the largest (2D
M2L by quarter-turn orbits, 3D M2L by reflection orbits), blob cores from far
wider than a leaf to points (both forms of the pair's factor and the line
between them), leaf counts around an item of targets.  Bar: 1e-12 of the
oracle's FMM, as everywhere on this path."""
import numpy as np
import pytest

import gpu_util as G
from paper_0905_2637_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL64 = 1e-12


@pytest.mark.parametrize("p", [1, 2, 3, 8, 13, 24, 39, 40])
@pytest.mark.parametrize("L,n", [(2, 300), (3, 2000), (5, 6000)])
def test_orders(orc, p, L, n):
    w = W.tiny(n, 100 + p, L=L, p=p, clustered_frac=0.3)
    u, v = G.run(w, "fp64")
    ur, vr = orc.fmm(w.x, w.y, w.gamma, w.domain, w.L, w.p, w.sigma)
    assert G.rel_l2(u, v, ur, vr) <= TOL64


@pytest.mark.parametrize("kappa", [1e-9, 1e-3, 0.5, 4.99, 5.0, 5.01, 20.0, 80.0, 1e5, 1e12])
def test_core_sizes(orc, kappa):
    # q = kappa rho^2 with rho^2 up to 8: the cells end at q = 40
    w = W.tiny(3000, 9, L=3, p=10, sigma=float(1 / 8 / np.sqrt(2 * kappa)), clustered_frac=0.2)
    u, v = G.run(w, "fp64")
    ur, vr = orc.fmm(w.x, w.y, w.gamma, w.domain, w.L, w.p, w.sigma)
    assert G.rel_l2(u, v, ur, vr) <= TOL64


def test_counts_around_an_item(orc):
    rng = np.random.default_rng(2)
    counts = rng.choice([0, 1, 2, 3, 4, 7, 8, 9, 15, 16, 17, 31, 32, 33, 48], size=(8, 8))
    pts = [((ix + rng.uniform(0, 1, c)) / 8, (iy + rng.uniform(0, 1, c)) / 8)
           for iy in range(8) for ix in range(8) for c in [int(counts[iy, ix])]]
    x, y = (np.concatenate(a) for a in zip(*pts))
    x[:5], y[:5] = x[5], y[5]  # coincident blobs
    w = W.Workload("items", x, y, rng.uniform(-1, 1, x.size), 0.02, W.UNIT_DOMAIN, 3, 17, "f64")
    u, v = G.run(w, "fp64")
    ur, vr = orc.fmm(w.x, w.y, w.gamma, w.domain, w.L, w.p, w.sigma)
    assert G.rel_l2(u, v, ur, vr) <= TOL64


@pytest.mark.parametrize("p", [1, 2, 5, 8, 9, 11, 16])
@pytest.mark.parametrize("L,n", [(2, 500), (3, 3000)])
def test_orders_3d(orc, p, L, n):
    import test_gpu_fmm3d as T
    w = W.tiny3d(n, 50 + p, L=L, p=p, clustered_frac=0.4)
    w.x[:3], w.y[:3], w.z[:3] = w.x[3], w.y[3], w.z[3]  # coincident charges
    rc, got = T._run(w, "fp64")
    assert rc == 0
    ref = orc.fmm3d(*w.as_f64(), w.domain, w.L, w.p)
    assert T._rel(got[0], ref[0]) <= TOL64 and T._field_rel(got, ref) <= TOL64
