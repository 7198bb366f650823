"""What a context holds from its creation: the tables its precision and depth
use, and no others (device memory of many contexts, less than one unused table
each), and every table that an option asks for later."""
import numpy as np
import pytest

import gpu_util as G
import test_gpu_fmm3d as T
from paper_0905_2637_gb300 import fmm3d
from paper_0905_2637_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _held(make, count=24):
    """Device bytes per context (allocations are carved from 2 MB pieces)."""
    torch = G.torch_cuda()
    for c in [make() for _ in range(count)]:  # module load, pools of streams and events
        c.close()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctxs = [make() for _ in range(count)]
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    for c in ctxs:
        c.close()
    return held / count


# 2D: the tensor cores' images exist up to p = 24 (5 MB there); a context that
# does not use them holds no more at 24 than at 25 (whose other tables are
# larger).
@pytest.mark.parametrize("precision,L", [("fp64", 10), ("mixed", 4)])
def test_2d_contexts_hold_their_own_tables(precision, L):
    _lib = G.lib()
    held = [_held(lambda: _lib.Context((0, 0, 1), L, p, 0.01, precision=precision)) for p in (24, 25)]
    assert held[0] <= held[1] + 2 * MB / 24, held  # (one 2 MB piece in all)


# 3D, p = 8: images 11.2 MB, matrices of the SIMT kernel 5.6 MB, orbits 1 MB.
@pytest.mark.parametrize("precision,L,bound", [("mixed", 5, 13 * MB), ("mixed", 3, 4 * MB),
                                               ("fp64", 5, 4 * MB)])
def test_3d_contexts_hold_their_own_tables(precision, L, bound):
    G.lib()
    assert _held(lambda: fmm3d.Context3D((0, 0, 0, 1), L, 8, precision=precision)) <= bound


def test_tables_asked_for_later(orc):
    # rows of tensor-core units, blocks at shallow levels, neither, in one context
    _lib = G.lib()
    w = W.tiny(20_000, 5, L=8, p=17, clustered_frac=0.3, dtype="f32")
    dev = G.to_dev((w.x, w.y, w.gamma))
    ur, vr = orc.fmm(*w.as_f64(), w.domain, w.L, w.p, w.sigma)
    ctx = _lib.Context(w.domain, w.L, w.p, w.sigma, precision="mixed", dtype="f32")
    for blocks in (0, 2, 1, 0):
        ctx.set_option(_lib.PETFMM_OPT_TC_BLOCKS, blocks)
        u, v = ctx.evaluate(*dev)
        assert ctx.sync() == 0
        assert G.rel_l2(u.cpu().numpy(), v.cpu().numpy(), ur, vr) <= 1e-5
    ctx.close()
    w = W.tiny3d(5000, 5, L=5, p=6, dtype="f32")
    rc, ref = T._run(w, "fp64")
    ctx = T._ctx(w, "mixed")
    for value in (0, 1, 2, 0):
        ctx.set_option(fmm3d.PETFMM3D_OPT_M2L_TC, value)
        rc, got = T._run(w, "mixed", ctx)
        assert rc == 0 and T._rel(got[0], ref[0]) <= 1e-5 and T._field_rel(got, ref) <= 1e-5
    ctx.close()
