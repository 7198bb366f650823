"""The task lists that evaluations launch (host only): contiguous, block-ordered
slices, and every level translated once -- M2L by tensor-core units or by
orbits, M2M upwards and L2L downwards level by level, the mixed path's top levels
in one launch."""
import numpy as np
import pytest

import __graft_entry__


@pytest.fixture(scope="module")
def lib():
    __graft_entry__.build()
    from paper_0905_2637_gb300 import _lib
    return _lib


def _instances(seed, k):
    rng = np.random.default_rng(seed)
    return [dict(domain=(0.0, 0.0, 1.0), levels=int(rng.integers(1, 11)), sigma=1e-3,
                 order=int(rng.choice([1, 8, 12, 17, 24, 25, 40])),
                 n=int(rng.integers(0, 50_000)) if i % 5 else 0) for i in range(k)]


PER_BLOCK = {0: 1024, 1: 256, 2: 256, 3: 256, 4: 256, 5: 32}  # units; the others: blocks


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("seed,k", [(1, 1), (2, 7), (3, 64), (4, 200)])
def test_launches_cover_every_level_once(lib, precision, seed, k):
    insts = _instances(seed, k)
    mixed = precision == 1
    lists = {}
    for row in lib.petfmm_debug_launches(precision, insts):
        lists.setdefault(int(row[0]), []).append([int(v) for v in row[1:]])
    for rid, rows in lists.items():
        per = PER_BLOCK.get(rid, 1)
        block = 0
        for _, _, units, block0 in rows:
            assert units > 0 and block0 == block
            block += -(-units // per)
    blocks = sum((2 ** (l - 1) // 8) * (2 ** (l - 1) // 16)
                 for it in insts if it["order"] <= 24 for l in range(5, min(it["levels"], 7) + 1))
    first = (5 if blocks >= 512 else 8) if mixed else 99
    # two runs of 128 (box, coefficient) pairs per block where there are enough
    def orbit_blocks(p, l, ni):
        rows = min(64, 128 * ni // p)
        return -(-4 ** (l - 1) // rows) * 4

    large = sum(orbit_blocks(it["order"], l, 2) for it in insts for l in range(2, it["levels"] + 1)
                if not (l >= first and it["order"] <= 24))
    ni = 2 if not mixed and large >= 608 else 1
    bottom = 4 if mixed else 2

    def of(rid, i):
        return {level: units for inst, level, units, _ in lists.get(rid, []) if inst == i}

    for i, it in enumerate(insts):
        L, p = it["levels"], it["order"]
        tensor = {l for l in range(first, L + 1)} if p <= 24 else set()
        assert of(6, i) == {}
        assert of(7, i) == {l: (2 ** (l - 1) // 8) * (2 ** (l - 1) // 16) for l in tensor}
        assert of(5, i) == {l: 4 ** l for l in tensor}
        assert of(8, i) == {l: orbit_blocks(p, l, ni) for l in range(2, L + 1) if l not in tensor}
        parents = max(1, min(32, 256 // p))
        shifts = {l: -(-4 ** l // parents) for l in range(bottom, L)}
        for first_id, order in ((100, [L - 1 - r for r in range(11)]), (200, [bottom + r for r in range(11)])):
            got = {}
            for r in range(11):
                level = of(first_id + r, i)
                assert set(level) <= {order[r]}
                got.update(level)
            assert got == shifts
        assert of(9, i) == ({min(L - 1, 3): 1} if mixed and max(x["levels"] for x in insts) >= 3 else {})
