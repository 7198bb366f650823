"""Contexts on a stream that does not wait for the legacy default stream: the
operator tables, uploaded when the context is made or inside an evaluation (a
new order, a new core width), are complete for the launches behind them."""
import numpy as np
import pytest

import gpu_util as G
import test_gpu_fmm3d as T
from paper_0905_2637_gb300 import fmm3d
from paper_0905_2637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_first_evaluations_of_new_tables(precision):
    _lib, torch = G.lib(), G.torch_cuda()
    w = W.tiny(3000, 4, L=3, p=17, clustered_frac=0.3)
    dev = G.to_dev((w.x, w.y, w.gamma))
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for p, sigma in ((17, 0.1), (30, 0.2), (9, 0.15), (23, 0.01), (12, 0.07)):
        with torch.cuda.stream(st):
            outs = [[torch.empty_like(dev[0]) for _ in range(2)] for _ in range(2)]
            ctx = _lib.Context((0, 0, 1), 2, 8, 0.01, precision=precision, dtype="f64", stream=st)
            for u, v in outs:  # a new order and core width inside the first call
                ctx.evaluate_batch([dict(domain=w.domain, levels=3, order=p, sigma=sigma, x=dev[0],
                                         y=dev[1], gamma=dev[2], u=u, v=v)])
            assert ctx.sync() == 0
            ctx.close()
        assert all(torch.equal(a, b) for a, b in zip(*outs))
        ref = [a.cpu().numpy() for a in outs[0]]
        alone = G.run(W.Workload("w", w.x, w.y, w.gamma, sigma, w.domain, 3, p, "f64"), precision)
        assert all(np.array_equal(a, b) for a, b in zip(ref, alone))


@pytest.mark.parametrize("precision,p", [("mixed", 8), ("mixed", 12), ("fp64", 8)])
def test_first_evaluation_3d(precision, p):
    torch = G.torch_cuda()
    w = W.tiny3d(2000, 4, L=2, p=p, dtype="f32")
    dev = G.to_dev((w.x, w.y, w.z, w.q))
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for _ in range(3):
        with torch.cuda.stream(st):
            out = [[torch.empty_like(dev[0]) for _ in range(4)] for _ in range(2)]
            ctx = fmm3d.Context3D(w.domain, w.L, p, precision=precision, dtype="f32", stream=st)
            for o in out:
                ctx.evaluate(*dev, out=o)
            assert ctx.sync() == 0
            ctx.close()
        assert all(torch.equal(a, b) for a, b in zip(*out))
    rc, ref = T._run(w, precision)
    assert rc == 0 and all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(out[0], ref))
