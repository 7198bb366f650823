"""The 3D mixed near field: leaf pairs summed pairwise (both leaves of at least
24 charges), the others one-sided, at the leaf counts where the work changes
form; against the FP64 path, and reproducible."""
import numpy as np
import pytest

import gpu_util as G
import test_gpu_fmm3d as T
from paper_0905_2637_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# around the pairwise limit, whole runs of 32, 64 and 128 targets with few left
# over, chunks of 32 sources with few left over, 2, 4 and 13 groups a leaf
COUNTS = [0, 0, 1, 5, 23, 24, 25, 31, 32, 33, 44, 52, 53, 63, 64, 65, 80, 81, 96, 97, 128, 129, 145,
          208, 385, 700]


def by_counts(counts, seed, dtype="f32"):
    rng = np.random.default_rng(seed)
    n = counts.shape[0]
    pts = [(np.array([ix, iy, iz]) + rng.uniform(0, 1, (int(counts[iz, iy, ix]), 3))) / n
           for iz in range(n) for iy in range(n) for ix in range(n)]
    pts = np.clip(np.concatenate(pts), 0.0, 1.0)
    t = np.float32 if dtype == "f32" else np.float64
    q = rng.uniform(-1, 1, len(pts))
    return W.Workload3D("counts", *(np.ascontiguousarray(pts[:, k], t) for k in range(3)),
                        q.astype(t), W.UNIT_CUBE, int(np.log2(n)), 8, dtype)


# The mixed path's bar: 1e-5 of the FP64 path (a dropped or doubled leaf pair
# shows at 1e-3 or more).
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_leaf_counts(seed, dtype):
    w = by_counts(np.random.default_rng(seed).choice(COUNTS, size=(4, 4, 4)), seed, dtype)
    rc, mixed = T._run(w, "mixed")
    assert rc == 0 and all(np.all(np.isfinite(a)) for a in mixed)
    rc, again = T._run(w, "mixed")
    assert all(np.array_equal(a, b) for a, b in zip(mixed, again))
    rc, ref = T._run(w, "fp64")
    assert T._rel(mixed[0], ref[0]) <= 1e-5 and T._field_rel(mixed, ref) <= 1e-5


def test_coincident_and_face_to_face():
    # coincident charges in a pairwise leaf, and charges on both sides of a
    # leaf face closer than FP32 resolves
    w = by_counts(np.full((2, 2, 2), 40), 7, "f64")
    w.x[:3], w.y[:3], w.z[:3] = w.x[3], w.y[3], w.z[3]
    w.x[10], w.y[10], w.z[10] = 0.5 - 1e-13, 0.25, 0.25
    w.x[11], w.y[11], w.z[11] = 0.5 + 1e-13, 0.25, 0.25
    rc, mixed = T._run(w, "mixed")
    assert rc == 0 and all(np.all(np.isfinite(a)) for a in mixed)
    rc, ref = T._run(w, "fp64")
    rest = np.setdiff1d(np.arange(w.n), [10, 11])
    assert T._rel(mixed[0][rest], ref[0][rest]) <= 1e-5


# One level: all eight leaves touch, so the FP64 result is the whole sum, up to
# the rounding of some thousand terms of mixed sign (n eps of the absolute sum,
# 1e-12 here; a dropped or doubled pair shows at 1e-5 or more).
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("seed", [1, 2, 3, 4])
def test_fp64_leaf_counts(seed, dtype):
    rng = np.random.default_rng(seed)
    counts = rng.choice(COUNTS + [2, 15, 16, 17, 127, 160, 256, 257], size=(2, 2, 2))
    w = by_counts(counts, seed, dtype)
    if w.n > 8:
        w.x[1], w.y[1], w.z[1] = w.x[0], w.y[0], w.z[0]  # a coincident pair
    rc, got = T._run(w, "fp64")
    assert rc == 0
    rc, again = T._run(w, "fp64")
    assert all(np.array_equal(a, b) for a, b in zip(got, again))
    x, y, z, q = (a.astype(np.float64) for a in (w.x, w.y, w.z, w.q))
    tol = 1e-12 if dtype == "f64" else 1e-7  # FP32 outputs round at 6e-8
    for i0 in range(0, w.n, 512):
        i = slice(i0, i0 + 512)
        d = [a[i, None] - a[None, :] for a in (x, y, z)]
        r2 = sum(a * a for a in d)
        same = r2 == 0
        r2[same] = 1.0
        p = np.where(same, 0.0, q[None, :] / np.sqrt(r2))
        for a, t in zip(got, [p] + [p / r2 * a for a in d]):
            assert np.all(np.abs(a[i] - t.sum(1)) <= tol * np.abs(t).sum(1) + 1e-30)


# M2L by reflection orbits, at the orders where the split over a block changes
# (one or several targets a group, 64, 128, 256 and 1,024 pairs), against the
# tensor-core kernel and the FP64 path: the mixed path's bar.
@pytest.mark.parametrize("L,p", [(2, 1), (2, 4), (2, 8), (3, 3), (3, 7), (3, 8), (4, 5), (2, 9),
                                 (3, 11), (3, 12), (4, 12), (3, 16)])
def test_orbit_m2l(L, p):
    from paper_0905_2637_gb300 import fmm3d
    w = W.tiny3d(6000 * 4 ** (L - 2), 50 + p, L=L, p=p, dtype="f32", clustered_frac=0.3)
    rc, got = T._run(w, "mixed")
    assert rc == 0
    rc, ref = T._run(w, "fp64")
    assert rc == 0
    assert T._rel(got[0], ref[0]) <= 1e-5 and T._field_rel(got, ref) <= 1e-5
    ctx = T._ctx(w, "mixed")
    ctx.set_option(fmm3d.PETFMM3D_OPT_M2L_TC, 1)
    rc, tc = T._run(w, "mixed", ctx)
    ctx.close()
    assert rc == 0 and T._field_rel(got, tc) <= 1e-5
