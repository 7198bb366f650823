"""The bounds-checked build on the files whose checks petfmm_debug_checks does
not report: expansions of the near field, M2M / L2L and M2L by orbits in both
precisions, batches of mixed depths, and the 3D path with hot, light and empty
leaves, pairwise and one-sided.  No recorded failure, each file in its own
word.  Runs in a child process, which loads the checked library."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import ctypes
import numpy as np, torch
from paper_0905_2637_gb300 import _lib, fmm3d
from paper_0905_2637_gb300 import workloads as W
assert _lib.LIB_PATH.endswith("libpetfmm_checked.so")
lines = (ctypes.c_uint32 * 7)()

def clean(what):
    n = _lib.load().petfmm_debug_checks_by_file(lines, 7)
    assert n == 7, n
    assert list(lines) == [0] * 7, (what, list(lines))

def dev(*a):
    return [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in a]

for precision in ("mixed", "fp64"):
    for L, p in ((3, 12), (5, 1), (6, 40)):
        for sigma in (0.5 ** L, 0.01):  # wide cores and narrow ones
            w = W.tiny(9000, L, L=L, p=p, clustered_frac=0.4, sigma=sigma)
            ctx = _lib.Context(w.domain, w.L, w.p, w.sigma, precision=precision, dtype=w.dtype)
            ctx.evaluate(*dev(w.x, w.y, w.gamma))
            assert ctx.sync() == 0
            ctx.close()
            clean((precision, L, p, sigma))
    insts = []
    ctx = _lib.Context((0, 0, 1), 2, 8, 0.01, precision=precision, dtype="f64")
    for i, (n, L) in enumerate(((0, 3), (1, 1), (700, 2), (5000, 6), (3000, 4))):
        w = W.tiny(n, i, L=L, p=8 + 3 * i, sigma=0.6 * 0.5 ** L)
        x, y, g = dev(w.x, w.y, w.gamma)
        insts.append(dict(domain=w.domain, levels=L, order=w.p, sigma=w.sigma, x=x, y=y, gamma=g,
                          u=torch.empty_like(x), v=torch.empty_like(x)))
    ctx.evaluate_batch(insts)
    assert ctx.sync() == 0
    ctx.close()
    clean((precision, "batch"))
    for L, p, n in ((2, 8, 3000), (3, 5, 9000), (3, 12, 3000), (5, 4, 40000)):
        w = W.tiny3d(n, L, L=L, p=p, clustered_frac=0.5)
        ctx = fmm3d.Context3D(w.domain, L, p, precision=precision, dtype=w.dtype)
        for pair_bytes in (1 << 34, 0):
            ctx.set_option(fmm3d.PETFMM3D_OPT_PAIR_BYTES, pair_bytes)
            ctx.evaluate(*dev(w.x, w.y, w.z, w.q))
            assert ctx.sync() == 0
            clean((precision, "3d", L, p, pair_bytes))
        ctx.close()
print("CHECKED-OK")
'''


def test_checked_build_reports_no_out_of_range_index_in_any_file():
    import __graft_entry__
    __graft_entry__.build()
    env = dict(os.environ, PETFMM_CHECKED="1", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "CHECKED-OK" in r.stdout
