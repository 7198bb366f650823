"""The FP64 path's own factors, value by value: g(q) = (1 - e^-q) / q from its
table and series step, 1 / sqrt(x) from its iteration, against extended
precision."""
import numpy as np
import pytest

import gpu_util as G
from paper_0905_2637_gb300 import fmm3d

pytestmark = pytest.mark.gpu

LD = np.longdouble
needs_longdouble = pytest.mark.skipif(np.finfo(LD).eps > 1e-18, reason="no extended precision")


def _ulps(got, ref):
    return np.abs(got.astype(LD) - ref) / np.spacing(np.abs(ref.astype(np.float64))).astype(LD)


# Rounded coefficients and Horner's steps, the argument's offset exact: 2 ulp;
# beyond q = 40 a rounded product and sum.
@needs_longdouble
def test_pair_factor_within_two_ulps():
    _lib = G.lib()
    rng = np.random.default_rng(1)
    edges = np.arange(0, 41 * 16) / 16.0
    q = np.concatenate([[0.0, 5e-324, 2.2250738585072014e-308, 1.7e308, 1e300, 4.4e307, 4.6e307], edges,
                        np.nextafter(edges[1:], 0), np.nextafter(edges, 100),
                        rng.uniform(0, 41, 400_000), rng.uniform(0, 0.07, 100_000),
                        10.0 ** rng.uniform(-300, 308, 100_000), rng.uniform(40, 2000, 100_000)])
    ctx = _lib.Context((0, 0, 1), 2, 4, 0.01, precision="fp64")
    got = ctx.debug_pair_factor(G.to_dev([q])[0])
    assert ctx.sync() == 0
    got = got.cpu().numpy()
    ctx.close()
    ql = q.astype(LD)
    ref = np.where(ql > 0, -np.expm1(-ql) / np.where(ql > 0, ql, 1), LD(1))
    assert np.all(np.isfinite(got)) and _ulps(got, ref).max() <= 2.0
    mixed = _lib.Context((0, 0, 1), 2, 4, 0.01, precision="mixed")
    with pytest.raises(_lib.PetfmmError):
        mixed.debug_pair_factor(G.to_dev([q])[0])
    mixed.close()


# e = 1 - x y^2 carries the rounding of x y (half of it reaches the result), and
# the last multiply-add rounds: 1.5 ulp.
@needs_longdouble
def test_rsqrt_within_one_and_a_half_ulps():
    G.lib()
    rng = np.random.default_rng(2)
    x = np.concatenate([[5e-324, 1e-310, 2.2250738585072014e-308, 1.7976931348623157e308, 1.0, 2.0, 4.0],
                        rng.uniform(1, 4, 400_000), 10.0 ** rng.uniform(-307, 308, 200_000),
                        np.nextafter(4.0 ** np.arange(-500, 500), 0), 4.0 ** np.arange(-500, 500)])
    ctx = fmm3d.Context3D((0, 0, 0, 1), 2, 4, precision="fp64", dtype="f64")
    got = ctx.debug_rsqrt(G.to_dev([x])[0])
    assert ctx.sync() == 0
    got = got.cpu().numpy()
    ctx.close()
    assert _ulps(got, 1 / np.sqrt(x.astype(LD))).max() <= 1.5
