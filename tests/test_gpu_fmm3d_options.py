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
