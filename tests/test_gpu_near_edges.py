"""The 2D near field at the edges of its arithmetic: pairs at subnormal
squared distances, coincident and lone blobs, infinite strengths, cores of
every width; against the FP64 oracle FMM or the exact value."""
import numpy as np
import pytest

import gpu_util as G
from paper_0905_2637_gb300 import workloads as W
from test_gpu_laplace import rel, run_laplace

pytestmark = pytest.mark.gpu


# A leaf centre of this domain lies at the coordinate origin, where FP32
# offsets far below the leaf's resolution elsewhere are kept.  1e-20 and 3e-20
# leaf widths: rho^2 is subnormal, of 17 bits or more, so its logarithm (about
# -92) is good to 1e-7.  Bar: the mixed path's 1e-5.
def test_laplace_pairs_at_subnormal_squared_distance(orc):
    rng = np.random.default_rng(1)
    x = np.concatenate([[0.0, 1e-20, 0.0, 0.3], rng.uniform(-1.5, 2.5, 60)])
    y = np.concatenate([[0.0, 0.0, 3e-20, 0.2], rng.uniform(-1.5, 2.5, 60)])
    w = W.Workload("close", x, y, rng.uniform(0.5, 1.0, x.size), 1.0, (-1.5, -1.5, 4.0), 2, 17, "f64")
    u, _ = run_laplace(w, precision="mixed")
    assert np.all(np.isfinite(u))
    assert rel(u, orc.laplace_fmm(w.x, w.y, w.gamma, w.domain, w.L, w.p)) <= 1e-5


# A charge has no potential of its own, nor has one at the same place: exactly
# zero, whatever the leaf width (its logarithm is a constant of the sum).
@pytest.mark.parametrize("width", [4.0, 1.0, 1e-6, 1e9])
def test_laplace_lone_and_coincident_charges_have_no_potential(width):
    x = np.full(5, 0.3 * width)
    for n in (1, 5):
        w = W.Workload("alone", x[:n], x[:n], np.arange(1.0, n + 1), 1.0, (0.0, 0.0, width), 1, 8, "f64")
        u, v = run_laplace(w, precision="mixed")
        assert np.all(u == 0.0) and np.all(v == 0.0)


# The busy times of the direct kernel (timing on) are kept by SM: a value for
# the SMs that have an entry, no effect on the result.
def test_busy_times_of_the_direct_kernel():
    w = W.tiny(40_000, 3, L=6, p=8, sigma=0.002)
    keep = []
    timed = G.run(w, "mixed", timing=True, ctx_out=keep)
    st = keep[0].stats()
    keep[0].close()
    assert 0.0 < st["p2p_load_balance"] <= 1.0
    assert all(np.array_equal(a, b) for a, b in zip(timed, G.run(w, "mixed")))


# The Laplace near field goes by work items in dense trees and by one thread per
# target in the others: a tree's form, and so its bits, are its own whatever
# the rest of its batch.
def test_laplace_batch_of_dense_and_sparse_trees_equals_alone():
    _lib, torch = G.lib(), G.torch_cuda()
    ws = [W.tiny(n, 20 + i, L=L, p=8, dtype="f32")
          for i, (n, L) in enumerate([(2000, 2), (4000, 6), (0, 3), (3000, 2), (900, 5), (1, 1)])]
    ctx = _lib.Context((0, 0, 1), 2, 8, 0.01, precision="mixed", dtype="f32", kernel="laplace")
    insts, outs = [], []
    for w in ws:
        x, y, g = G.to_dev((w.x, w.y, w.gamma))
        outs.append((torch.empty_like(x), torch.empty_like(x)))
        insts.append(dict(domain=w.domain, levels=w.L, order=w.p, sigma=w.sigma, x=x, y=y, gamma=g,
                          u=outs[-1][0], v=outs[-1][1]))
    ctx.evaluate_batch(insts)
    assert ctx.sync() == 0
    ctx.close()
    for w, (u, v) in zip(ws, outs):
        if w.n:
            assert np.array_equal(u.cpu().numpy().astype(np.float64), run_laplace(w, precision="mixed")[0])


# Cores down to 1e-300: point vortices to every bit of the FP64 path, whatever
# 1 / 2 sigma^2 overflows to.  The oracle's FMM in the unit square, at a core far
# below every distance (the tree scales with a power of two exactly).
@pytest.mark.parametrize("sigma,width", [(1e-100, 1.0), (1e-150, 1.0), (1e-160, 1.0), (1e-300, 1.0),
                                         (1e-160, 2.0 ** 133), (1e-200, 2.0 ** -133),
                                         (1e-260, 2.0 ** -133)])
def test_fp64_point_vortices(orc, sigma, width):
    w = W.tiny(1500, 8, L=3, p=12, clustered_frac=0.2)
    w.x[:3], w.y[:3] = w.x[3], w.y[3]  # coincident: nothing from one another
    ur, vr = orc.fmm(w.x, w.y, w.gamma, w.domain, w.L, w.p, 1e-9)
    w = W.Workload("points", w.x * width, w.y * width, w.gamma, sigma, (0.0, 0.0, width), 3, 12, "f64")
    u, v = G.run(w, "fp64")
    assert G.rel_l2(u * width, v * width, ur, vr) <= 1e-12


# Cores far narrower than a leaf, down to points, in every form of the mixed
# near field: the polynomial's coefficients in rho^2 grow as kappa^5 and leave
# FP32's range, those in q do not.  Bar: the mixed path's 1e-5.
@pytest.mark.parametrize("form", [0, 1, 2])
@pytest.mark.parametrize("sigma", [1e-3, 3e-5, 1e-5, 1e-6, 1e-9, 1e-13, 1e-20, 1e-100, 1e-300])
def test_mixed_narrow_cores(orc, sigma, form):
    w = W.tiny(3000, 8, L=3, p=12, clustered_frac=0.2, sigma=sigma)
    w.x[:3], w.y[:3] = w.x[3], w.y[3]  # coincident: nothing from one another
    u, v = G.run(w, "mixed", options={G.lib().PETFMM_OPT_P2P_PAIRS: form})
    ur, vr = orc.fmm(w.x, w.y, w.gamma, w.domain, w.L, w.p, max(sigma, 1e-9))
    assert np.all(np.isfinite(u)) and G.rel_l2(u, v, ur, vr) <= 1e-5


# The pair factor alone, trees of two blobs, q = r^2 / 2 sigma^2 over the line
# between its two forms.  FP32's bound per bin of q: the polynomial's 11e-8 rms or
# the exponential form's 7e-8, and some six roundings of 3.4e-8 rms: 14e-8.
@pytest.mark.parametrize("kappa", [3.5, 27.0])
def test_pair_factor_keeps_fp32_accuracy(kappa):
    _lib, torch = G.lib(), G.torch_cuda()
    rng = np.random.default_rng(2)
    edges = np.array([0.02, 0.05, 0.07, 0.1, 0.15, 0.2, 0.3, 0.4, 0.5, 0.6, 0.7, 0.8, 1.0, 1.5])
    per = 160
    q = np.concatenate([rng.uniform(a, b, per) for a, b in zip(edges, edges[1:])])
    sigma = float(0.5 / np.sqrt(2 * kappa))  # leaves of 1/2
    r, th = sigma * np.sqrt(2 * q), rng.uniform(0, 2 * np.pi, q.size)
    ax, ay = rng.uniform(0.45, 0.55, (2, q.size))
    x = np.stack([ax, ax + r * np.cos(th)], 1).astype(np.float32)
    y = np.stack([ay, ay + r * np.sin(th)], 1).astype(np.float32)
    dx, dy, g = *G.to_dev((x, y)), torch.ones(q.size, 2, device="cuda")
    u, v = torch.empty_like(dx), torch.empty_like(dx)
    ctx = _lib.Context((0, 0, 1), 1, 4, 0.01, precision="mixed", dtype="f32")
    ctx.evaluate_batch([dict(domain=(0.0, 0.0, 1.0), levels=1, order=4, sigma=sigma, x=dx[i], y=dy[i],
                             gamma=g[i], u=u[i], v=v[i]) for i in range(q.size)])
    assert ctx.sync() == 0
    ctx.close()
    ex, ey = (a[:, 0].astype(np.float64) - a[:, 1] for a in (x, y))
    r2 = ex ** 2 + ey ** 2
    f = -np.expm1(-r2 / (2 * sigma ** 2)) / (2 * np.pi * r2)
    err = np.hypot(u[:, 0].cpu().numpy() + f * ey, v[:, 0].cpu().numpy() - f * ex) / (f * np.sqrt(r2))
    rms = np.sqrt((err.reshape(-1, per) ** 2).mean(1))
    assert np.all(rms <= 2e-7), dict(zip(edges.round(2), rms))


# A blob of infinite strength moves the others, not itself nor one at its place.
def test_fp64_infinite_strength_adds_nothing_to_itself():
    x = np.array([0.3, 0.3, 0.31, 0.8])
    w = W.Workload("inf", x, x[::-1].copy(), np.array([np.inf, 2.0, 1.0, -1.0]), 0.05, (0, 0, 1.0), 1, 4,
                   "f64")
    w.y[:2] = 0.4
    u, v = G.run(w, "fp64")
    d = np.hypot(w.x[:, None] - w.x, w.y[:, None] - w.y)
    f = np.where(d > 0, -np.expm1(-d ** 2 / (2 * w.sigma ** 2)) / (2 * np.pi * np.where(d > 0, d, 1) ** 2), 0)
    for i in (0, 1):
        k = [2, 3]  # the blobs elsewhere
        want = (-(f[i, k] * w.gamma[k] * (w.y[i] - w.y[k])).sum(), (f[i, k] * w.gamma[k] * (w.x[i] - w.x[k])).sum())
        assert np.allclose((u[i], v[i]), want, rtol=1e-12, atol=0)
    assert np.all(np.isinf(u[2:])) and np.all(np.isinf(v[2:]))
