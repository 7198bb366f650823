"""The mixed path's near field by expansions (blob cores wide against a leaf):
against the FP64 oracle FMM at leaf counts around the limits between direct
leaf pairs and expansions, for every degree, alone and in a batch."""
import numpy as np
import pytest

import gpu_util as G
from paper_0905_2637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def wide_core(kappa, counts, seed, dtype="f32"):
    """Blobs with the given counts per leaf [iy, ix]; sigma from kappa = w^2 / 2 sigma^2."""
    rng = np.random.default_rng(seed)
    n = counts.shape[0]
    xs, ys = [], []
    for iy in range(n):
        for ix in range(n):
            c = int(counts[iy, ix])
            xs.append((ix + rng.uniform(0.001, 0.999, c)) / n)
            ys.append((iy + rng.uniform(0.001, 0.999, c)) / n)
    x, y = np.concatenate(xs), np.concatenate(ys)
    g = rng.uniform(-1.0, 1.0, x.size)
    t = np.float32 if dtype == "f32" else np.float64
    return W.Workload("wide-core", x.astype(t), y.astype(t), g.astype(t),
                      float(1.0 / n / np.sqrt(2 * kappa)), W.UNIT_DOMAIN, int(np.log2(n)), 12, dtype)


# The expansions reproduce a pair to 1.2e-7 of the kernel's largest value and
# FP32 sums add a few roundings; the mixed path's bar against the FP64 FMM is
# 1e-5, and directed pairs (each factor within 2.5e-6) stay within it too.
@pytest.mark.parametrize("kappa", [1e-4, 0.119, 0.169, 0.25, 0.49, 0.9, 1.9])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_counts_around_the_limits(orc, kappa, dtype):
    rng = np.random.default_rng(3)
    counts = rng.choice([0, 0, 1, 2, 15, 16, 17, 23, 24, 31, 33, 42, 43, 64, 129, 1900], size=(8, 8))
    w = wide_core(kappa, counts, 5, dtype)
    u1, v1 = G.run(w, "mixed")
    assert np.all(np.isfinite(u1)) and np.all(np.isfinite(v1))
    ur, vr = orc.fmm(w.x, w.y, w.gamma, w.domain, w.L, w.p, w.sigma)
    e1 = G.rel_l2(u1, v1, ur, vr)
    u0, v0 = G.run(w, "mixed", options={G.lib().PETFMM_OPT_P2P_PAIRS: 0})
    e0 = G.rel_l2(u0, v0, ur, vr)
    assert e1 <= 1e-5 and e1 <= e0 + 1e-6, (e1, e0)


@pytest.mark.parametrize("n,L", [(1, 1), (1, 3), (2, 1), (40, 1), (300, 2), (5000, 1), (70_000, 2)])
def test_small_and_shallow(orc, n, L):
    w = W.tiny(n, 7, L=L, p=8, sigma=0.9 / (1 << L), dtype="f32")
    u1, v1 = G.run(w, "mixed")
    ur, vr = orc.fmm(w.x, w.y, w.gamma, w.domain, w.L, w.p, w.sigma)
    assert G.rel_l2(u1, v1, ur, vr) <= 1e-5


def test_batch_of_degrees_equals_alone():
    # instances of every degree, and one that sums pairs, interleaved in the
    # occupied list of one batch: each bit for bit its result alone
    _lib = G.lib()
    torch = G.torch_cuda()
    rng = np.random.default_rng(9)
    ws = [wide_core(k, rng.choice([0, 3, 20, 70, 300], size=(4, 4)), i)
          for i, k in enumerate([0.119, 0.119, 0.3, 8.0, 0.8, 0.15, 1.7])]
    ctx = _lib.Context((0, 0, 1), 2, 8, 0.01, precision="mixed", dtype="f32")
    insts, outs = [], []
    for w in ws:
        x, y, g = G.to_dev((w.x, w.y, w.gamma))
        u, v = torch.empty_like(x), torch.empty_like(x)
        insts.append(dict(domain=w.domain, levels=w.L, order=w.p, sigma=w.sigma, x=x, y=y, gamma=g,
                          u=u, v=v))
        outs.append((u, v))
    for _ in range(2):
        ctx.evaluate_batch(insts)
    assert ctx.sync() == 0
    ctx.close()
    for w, (u, v) in zip(ws, outs):
        ua, va = G.run(w, "mixed")
        assert np.array_equal(u.cpu().numpy(), ua) and np.array_equal(v.cpu().numpy(), va)


# A near-field tolerance below what the expansions keep (4.2e-7 of the kernel's
# largest value, tests/test_smooth_operator.py) is kept by pair sums.  No leaf
# has the 32 blobs of the pair kernel, so those are option 1's, bit for bit.
@pytest.mark.parametrize("tol,summed", [(100, True), (419, True), (420, False), (2500, False)])
def test_small_tolerances_sum_pairs(tol, summed):
    _lib = G.lib()
    w = wide_core(0.119, np.random.default_rng(1).integers(16, 32, (8, 8)), 2)
    got = [G.run(w, "mixed", options={_lib.PETFMM_OPT_NEAR_TOL: tol, _lib.PETFMM_OPT_P2P_PAIRS: form})
           for form in (2, 1)]
    assert np.array_equal(got[0][0], got[1][0]) == summed
    assert np.array_equal(got[0][1], got[1][1]) == summed


def test_first_evaluations_on_several_threads():
    # contexts of their own on threads of their own, all at their first wide core
    import threading
    _lib, torch = G.lib(), G.torch_cuda()
    ws = [wide_core(k, np.full((4, 4), 60), i) for i, k in enumerate([0.1, 0.3, 0.8, 1.7] * 2)]
    dev = [G.to_dev((w.x, w.y, w.gamma)) for w in ws]
    torch.cuda.synchronize()
    out, go = [None] * len(ws), threading.Barrier(len(ws))

    def work(i):
        w, st = ws[i], torch.cuda.Stream()
        go.wait()
        with torch.cuda.stream(st):
            ctx = _lib.Context(w.domain, w.L, w.p, w.sigma, precision="mixed", dtype="f32", stream=st)
            u, v = ctx.evaluate(*dev[i])
            assert ctx.sync() == 0
            ctx.close()
        out[i] = u.cpu().numpy(), v.cpu().numpy()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(ws))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for w, got in zip(ws, out):
        ref = G.run(w, "mixed")
        assert got is not None and all(np.array_equal(a, b) for a, b in zip(got, ref))
