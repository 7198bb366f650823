"""3D near field with leaves so full that a leaf pair would be a large part of
the whole: such pairs are shared out one-sided over many warps, the others of
the same tree stay pairwise."""
import numpy as np
import pytest

import test_gpu_fmm3d as T
from paper_0905_2637_gb300 import fmm3d
from paper_0905_2637_gb300 import workloads as W
from test_gpu_near3d import by_counts

pytestmark = pytest.mark.gpu

# One level: all leaves touch, so the FP64 result is the whole sum, up to the
# rounding of some thousand terms of mixed sign (n eps of the absolute sum, 1e-12
# here; a dropped or doubled leaf pair shows at 1e-5 or more).  Mixed: 1e-5.
COUNTS = [[3000, 40, 0, 700, 1, 90, 33, 200], [4000, 0, 0, 0, 0, 0, 0, 0], [1500, 1500, 0, 7, 0, 25, 0, 0],
          [2500, 1, 64, 64, 64, 64, 64, 65]]


@pytest.mark.parametrize("counts", COUNTS)
def test_hot_leaves(counts):
    w = by_counts(np.array(counts).reshape(2, 2, 2), 3, "f64")
    w.x[1], w.y[1], w.z[1] = w.x[0], w.y[0], w.z[0]  # a coincident pair
    rc, got = T._run(w, "fp64")
    assert rc == 0
    rc, again = T._run(w, "fp64")
    assert all(np.array_equal(a, b) for a, b in zip(got, again))
    for i0 in range(0, w.n, 512):
        i = slice(i0, i0 + 512)
        d = [a[i, None] - a[None, :] for a in (w.x, w.y, w.z)]
        r2 = sum(a * a for a in d)
        same = r2 == 0
        r2[same] = 1.0
        p = np.where(same, 0.0, w.q[None, :] / np.sqrt(r2))
        for a, t in zip(got, [p] + [p / r2 * a for a in d]):
            assert np.all(np.abs(a[i] - t.sum(1)) <= 1e-12 * np.abs(t).sum(1) + 1e-30)
    rc, mixed = T._run(w, "mixed")
    assert rc == 0
    rc, again = T._run(w, "mixed")
    assert all(np.array_equal(a, b) for a, b in zip(mixed, again))
    assert T._rel(mixed[0], got[0]) <= 1e-5 and T._field_rel(mixed, got) <= 1e-5


# All charges in one leaf: 2.7e8 ordered pairs.  Shared by every SM the FP64 sums
# take about 10 ms (18 operations a pair, two lanes a cycle and SM) and the FP32
# ones 1 ms; one warp alone takes 1.6 s and 60 ms.
@pytest.mark.parametrize("precision,limit_ms", [("fp64", 100.0), ("mixed", 10.0)])
def test_one_full_leaf_is_shared_by_the_whole_gpu(precision, limit_ms):
    rng = np.random.default_rng(1)
    n = 16384
    pts = 0.3 + 0.1 * rng.uniform(0, 1, (3, n))
    w = W.Workload3D("one leaf", *pts, rng.uniform(-1, 1, n), W.UNIT_CUBE, 2, 4, "f64")
    ctx = T._ctx(w, precision)
    ctx.set_option(fmm3d.PETFMM3D_OPT_TIMING, 1)
    for _ in range(3):
        rc, _ = T._run(w, precision, ctx)
        assert rc == 0
    near = ctx.stage_times()["near"]
    ctx.close()
    assert near <= limit_ms, near
