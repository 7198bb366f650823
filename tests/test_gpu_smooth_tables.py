"""Operators of the near field by expansions, made on the device when a core
width is first met: against the host's, kept and replaced, under graph replay."""
import time

import numpy as np
import pytest

import gpu_util as G
from paper_0905_2637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _insts(ws, dtype="f32"):
    torch = G.torch_cuda()
    insts, outs = [], []
    for w in ws:
        x, y, g = G.to_dev((w.x, w.y, w.gamma))
        outs.append((torch.empty_like(x), torch.empty_like(x)))
        insts.append(dict(domain=w.domain, levels=w.L, order=w.p, sigma=w.sigma, x=x, y=y, gamma=g,
                          u=outs[-1][0], v=outs[-1][1]))
    return insts, outs


def _wide(kappa, n, seed, L=1):
    return W.tiny(n, seed, L=L, p=4, sigma=float(0.5 ** L / np.sqrt(2 * kappa)), dtype="f32")


def _same(_lib, table, kappa):
    n, op = table
    nh, ref = _lib.petfmm_debug_smooth_operators(kappa)
    # entries of order one, made in FP64 and rounded: an FP32 rounding apart
    assert n == nh and np.all(np.abs(op - ref) <= 6e-8 * np.abs(ref) + 1e-10)


@pytest.mark.parametrize("graph", [0, 1])
def test_tables_match_the_host_and_give_the_results_alone(graph):
    # 200 widths of every degree in one batch (several launches, more than the
    # smallest buffer), then others in the same context, then the first again
    _lib = G.lib()
    rng = np.random.default_rng(4)
    kappas = [np.concatenate([rng.uniform(0.01, 1.95, 196), [0.17, 0.5, 1.04, 1.95]]),
              rng.uniform(0.01, 1.95, 3)]
    ctx = _lib.Context((0, 0, 1), 2, 8, 0.01, precision="mixed", dtype="f32")
    ctx.set_option(_lib.PETFMM_OPT_GRAPH, graph)
    for which in (0, 1, 0, 1):
        ws = [_wide(k, 400, i) for i, k in enumerate(kappas[which])]
        insts, outs = _insts(ws)
        for _ in range(2):
            ctx.evaluate_batch(insts)
        assert ctx.sync() == 0
        for i in range(0, len(ws), 7):
            k = (0.5 / ws[i].sigma) ** 2 / 2
            _same(_lib, ctx.debug_smooth_table(i), k)
            ua, va = G.run(ws[i], "mixed")
            assert np.array_equal(outs[i][0].cpu().numpy(), ua) and np.array_equal(outs[i][1].cpu().numpy(), va)
    ctx.close()


def test_small_trees_have_no_tables():
    # too few blobs for any leaf pair to go by expansions
    _lib = G.lib()
    ctx = _lib.Context((0, 0, 1), 2, 8, 0.01, precision="mixed", dtype="f32")
    ws = [_wide(0.1, 12, 1), _wide(0.1, 400, 2)]
    insts, _ = _insts(ws)
    ctx.evaluate_batch(insts[:1])
    assert ctx.sync() == 0 and ctx.debug_smooth_table(0) == (0, None)
    ctx.evaluate_batch(insts)
    assert ctx.sync() == 0 and ctx.debug_smooth_table(1)[0] == 8
    ctx.close()


# A time step whose domain is refitted meets a new width: some 10 us of device
# work, where the tables made on the host took 0.65 to 1.6 ms.
def test_a_new_width_costs_little():
    _lib, torch = G.lib(), G.torch_cuda()
    w = _wide(1.2, 4000, 3, L=3)
    insts, _ = _insts([w])
    ctx = _lib.Context((0, 0, 1), 2, 8, 0.01, precision="mixed", dtype="f32")

    def per_call(sigmas):
        times = []
        for s in sigmas:
            t = time.perf_counter()
            ctx.evaluate_batch([dict(insts[0], sigma=float(s))])
            assert ctx.sync() == 0
            times.append(time.perf_counter() - t)
        return float(np.median(times))

    per_call([w.sigma] * 5)
    same = per_call([w.sigma] * 60)
    new = per_call(w.sigma * (1 + 1e-4 * np.arange(1, 61)))
    ctx.close()
    assert new - same <= 2.5e-4, (new, same)
