"""The 3D options: which values are taken, and that each can be left again."""
import numpy as np
import pytest

import gpu_util as G
import test_gpu_fmm3d as T
from paper_0905_2637_gb300 import fmm3d
from paper_0905_2637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _eval(ctx, w):
    out = ctx.evaluate(*G.to_dev((w.x, w.y, w.z, w.q)))
    assert ctx.sync() == 0
    return [a.cpu().numpy() for a in out]


def test_m2l_option_returns_to_its_default():
    w = W.tiny3d(6000, 3, L=3, p=8, dtype="f32")
    ctx = T._ctx(w, "mixed")
    first = _eval(ctx, w)
    others = []
    for value in (1, 0):
        ctx.set_option(fmm3d.PETFMM3D_OPT_M2L_TC, value)
        others.append(_eval(ctx, w))
    ctx.set_option(fmm3d.PETFMM3D_OPT_M2L_TC, 2)
    again = _eval(ctx, w)
    for value in (-1, 3):
        with pytest.raises(Exception):
            ctx.set_option(fmm3d.PETFMM3D_OPT_M2L_TC, value)
    ctx.close()
    assert all(np.array_equal(a, b) for a, b in zip(first, again))
    for o in others:  # (three different kernels at three levels)
        assert not np.array_equal(first[0], o[0]) and T._rel(first[0], o[0]) <= 1e-5


# Every leaf pair from both sides (PETFMM3D_OPT_PAIR_BYTES = 0), at many charges
# with hot, light and empty leaves: within the path's rounding of the default
# (FP64: 1e-12, mixed: two results each within 1e-5 of the FP64 path), and the
# default's bits again afterwards.
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
def test_pairs_from_both_sides(precision, tol):
    # (an even tree of enough pairs has pairwise sums; in the others it depends on
    # their weights)
    for w, even in ((W.tiny3d(60_000, 5, L=3, p=8), True),
                    (W.tiny3d(20_000, 5, L=3, p=8, clustered_frac=0.5), False),
                    (W.tiny3d(3000, 6, L=1, p=4, clustered_frac=0.2), False)):
        ctx = T._ctx(w, precision)
        first = _eval(ctx, w)
        ctx.set_option(fmm3d.PETFMM3D_OPT_PAIR_BYTES, 0)
        both = _eval(ctx, w)
        assert all(np.array_equal(a, b) for a, b in zip(both, _eval(ctx, w)))
        ctx.set_option(fmm3d.PETFMM3D_OPT_PAIR_BYTES, 1 << 34)
        again = _eval(ctx, w)
        with pytest.raises(Exception):
            ctx.set_option(fmm3d.PETFMM3D_OPT_PAIR_BYTES, -1)
        ctx.close()
        assert not (even and np.array_equal(first[0], both[0]))
        assert all(np.array_equal(a, b) for a, b in zip(first, again))
        assert T._rel(both[0], first[0]) <= tol and T._field_rel(both, first) <= tol


def _fill(torch, leave):
    """All free device memory but `leave` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


# Where the memory for pairwise sums cannot be had beside the needed buffers, the
# call works without it: (a) a new context, room for that memory but not for
# all else besides; (b) a context that holds it and grows.
def test_evaluation_works_without_room_for_pairwise_sums():
    torch = G.torch_cuda()
    n, mb = 4_000_000, 1 << 20
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    big = [torch.rand(3 * n // 2, generator=g, device="cuda") for _ in range(4)]
    small = [t[:n] for t in big]
    out = {len(a[0]): [torch.empty_like(a[0]) for _ in range(4)] for a in (small, big)}

    def run(ctx, args):
        ctx.evaluate(*args, out=out[len(args[0])])
        assert ctx.sync() == 0
        return [t.clone() for t in out[len(args[0])]]

    def ctx(pair_bytes=None):
        c = fmm3d.Context3D((0, 0, 0, 1.0), 5, 4)
        if pair_bytes is not None:
            c.set_option(fmm3d.PETFMM3D_OPT_PAIR_BYTES, pair_bytes)
        return c

    c = ctx(0)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    want, want_big = run(c, small), None
    needed = before - torch.cuda.mem_get_info()[0] - 4 * 4 * n  # (less the copies of the results)
    want_big = run(c, big)
    c.close()
    slots, own = 416 * n, 16 * n
    c = ctx()
    hold = _fill(torch, needed + slots - own // 2)
    ctx_out = out[n]
    c.evaluate(*small, out=ctx_out)
    assert c.sync() == 0
    del hold
    torch.cuda.empty_cache()
    assert all(torch.equal(a, b) for a, b in zip(ctx_out, want))
    # (b)
    c.set_option(fmm3d.PETFMM3D_OPT_PAIR_BYTES, 1 << 34)
    paired = run(c, small)
    assert not torch.equal(paired[0], want[0])
    hold = _fill(torch, 64 * mb)
    c.evaluate(*big, out=out[len(big[0])])
    assert c.sync() == 0
    del hold
    torch.cuda.empty_cache()
    assert all(torch.equal(a, b) for a, b in zip(out[len(big[0])], want_big))
    c.close()
