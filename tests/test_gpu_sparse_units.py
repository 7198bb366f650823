"""Block units of the tensor-core M2L with few occupied cells: a source class
that only one or two cells hold must never be dropped (the mask of the classes
is cleared before any thread sets a bit of it)."""
import numpy as np
import pytest
import torch

from paper_0905_2637_gb300 import _lib

pytestmark = pytest.mark.gpu


def test_sparse_units_give_the_same_bits_every_time():
    # eight clusters wide enough that most units of 16 x 32 leaves hold a few
    # dozen blobs, some only six to ten
    rng = np.random.default_rng(5)
    n = 60_000
    c = rng.uniform(0.2, 0.8, (8, 2))[rng.integers(0, 8, n)]
    x, y = np.clip(c + 0.05 * rng.standard_normal((n, 2)), 0, 1).T.astype(np.float32)
    g = (rng.standard_normal(n) / n).astype(np.float32)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, y, g)]
    ctx = _lib.Context((0, 0, 1), 10, 17, 0.002, precision="mixed", dtype="f32")
    u, v = ctx.evaluate(*dev)
    assert ctx.sync() == 0
    first = u.clone(), v.clone()
    for _ in range(300):
        ctx.evaluate(*dev, u, v)
        assert ctx.sync() == 0
        assert torch.equal(u, first[0]) and torch.equal(v, first[1])
    ctx.close()
    ref = _lib.Context((0, 0, 1), 10, 17, 0.002, precision="fp64", dtype="f32")
    ru, rv = ref.evaluate(*dev)
    assert ref.sync() == 0
    ref.close()
    d = (u.double() - ru.double()) ** 2 + (v.double() - rv.double()) ** 2
    assert float((d.sum() / (ru.double() ** 2 + rv.double() ** 2).sum()).sqrt()) <= 1e-5
