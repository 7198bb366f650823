"""Host operators of the near field by expansions (blob cores wide against a
leaf): against the pair velocity of Eq. 8 in FP64 over the near domain, at both
ends of every degree's range."""
import numpy as np
import pytest
from numpy.polynomial import legendre

from paper_0905_2637_gb300 import _lib


@pytest.mark.parametrize("kappa,degree", [
    (1e-4, 8), (0.17, 8), (0.171, 10), (0.50, 10), (0.501, 12), (1.04, 12), (1.041, 14), (1.95, 14)])
def test_expansion_reproduces_the_pair_velocity(kappa, degree):
    n, op = _lib.petfmm_debug_smooth_operators(kappa)
    assert n == degree and np.all(np.isfinite(op))
    rng = np.random.default_rng(11)
    corners = 0.5 * np.array([(x, y) for x in (-1, 0, 1) for y in (-1, 0, 1)])
    tau = np.concatenate([corners, rng.uniform(-0.5, 0.5, (200, 2))])
    src = np.concatenate([-corners, rng.uniform(-0.5, 0.5, (200, 2))])
    terms = [(a, b) for b in range(n + 1) for a in range(n + 1 - b)]
    px, py = (legendre.legvander(2 * src[:, k], n) for k in (0, 1))
    mom = np.array([px[:, a] * py[:, b] for a, b in terms])
    tx, ty = (np.vander(2 * tau[:, k], n + 1, increasing=True) for k in (0, 1))
    z = np.zeros(len(tau))
    gx = np.array([2 * a * tx[:, a - 1] * ty[:, b] if a else z for a, b in terms])
    gy = np.array([2 * b * tx[:, a] * ty[:, b - 1] if b else z for a, b in terms])
    top, err = 0.0, 0.0
    for o in range(9):
        d = tau[:, None, :] - src[None, :, :] - np.array([o % 3 - 1, o // 3 - 1])
        q = kappa * (d ** 2).sum(-1)
        g = np.where(q > 0, -np.expm1(-q) / np.where(q > 0, q, 1), 1.0)
        top = max(top, np.abs(d * g[..., None]).max())
        loc = op[o].astype(np.float64).T @ mom
        err = max(err, np.abs(gx.T @ loc - d[..., 0] * g).max(),
                  np.abs(gy.T @ loc - d[..., 1] * g).max())
    # the projection's own error, and the FP32 rounding of M entries per row
    # and column (relative 6e-8 each, adding as a random walk)
    assert err <= (1.2e-7 + 3e-7) * top


def test_narrow_cores_sum_pairs():
    for kappa in (1.951, 8.0, 100.0):
        assert _lib.petfmm_debug_smooth_operators(kappa) == (0, None)
