"""Bulk merge into a table whose cells are still in sorted order (two runs are
merged, the batch alone is sorted), and the bulk build's sort at the edges of
its tiles.  The layout is deterministic: cells equal the oracle's bit for bit.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import codes_buf, to_dev, to_np_u8, to_np_u64, vals_buf

pytestmark = pytest.mark.gpu

MAX = (1 << 64) - 1


def _cells(t):
    return to_np_u64(t.cells()).reshape(-1, 2)


@pytest.mark.parametrize("log2c,n,m,erase,kw", [
    (13, 4096, 1, 0, {}),                                      # one pair; 4096 cells: one tile of the merge twice over
    (13, 4096, 2048, 0, {}),                                   # the largest batch that goes this way
    (13, 4096, 2049, 0, {}),                                   # one more: the general way
    (16, 50_000, 12_345, 0, {}),                               # ragged tiles, load near 0.9, a dense write
    (16, 30_000, 9_000, 7_000, {}),                            # tombstones between the live cells
    (18, 20_000, 3_001, 0, {}),                                # fewer than an eighth of the cells: a sparse write
    (15, 16_000, 8_000, 100, {"growable": True}),              # grows to 2^16
    (16, 30_000, 10_000, 0, {"full": True}),                   # keys 0 / ~0 to the special slots
    (16, 30_000, 10_000, 0, {"reserved": True}),               # keys 0 / ~0 skipped
])
def test_merge_into_sorted_table(cuda_lib, oracle_mod, log2c, n, m, erase, kw):
    growable, full = kw.get("growable", False), kw.get("full", False)
    rng = np.random.default_rng(n + m)
    pool = W.uniform_keys(n + m, start=n * 1000, seed=71)
    keys, vals = pool[:n], rng.integers(1, 1 << 62, n).astype(np.uint64)
    t = cuda_lib.Table(1 << log2c, growable=growable)
    t.set_config(full_key_space=int(full))
    o = oracle_mod.OracleTable(1 << log2c, growable=growable, alpha=0.5, full_key_space=full)
    t.build(to_dev(keys), to_dev(vals))
    assert o.build(keys, vals) == 0
    if erase:
        gone = keys[rng.permutation(n)[:erase]]
        t.erase(to_dev(gone))
        o.erase(gone)
    for _ in range(2):  # the second merge goes into the first one's cells
        bk = pool[rng.integers(0, n + m, m)]
        bk[: m // 8] = bk[0]  # one key many times
        if full or kw.get("reserved"):
            bk[rng.integers(0, m, 3)] = [0, MAX, 0]
        bv = rng.integers(1, 1 << 62, m).astype(np.uint64)
        t.merge(to_dev(bk), to_dev(bv))
        assert o.merge(bk, bv) in (0, 1)
        assert np.array_equal(_cells(t), o.cells())
        assert t.size() == (o.live, o.nonempty, o.capacity)
    if full:
        q = np.array([0, MAX], np.uint64)
        vo, fo = vals_buf(2), codes_buf(2)
        t.find(to_dev(q), vo, fo)
        ev, ef = o.find(q)
        assert np.array_equal(to_np_u8(fo), ef) and np.array_equal(to_np_u64(vo), ev)


def test_merge_into_sorted_table_that_wraps(cuda_lib, oracle_mod):
    # keys homed in the last cells: the build's tail wraps to the first cells,
    # which are then out of order, and a batch homed there too
    log2c = 12
    cand = W.uniform_keys(400_000, start=0, seed=72)
    h = oracle_mod.homes(cand, log2c)
    tail = cand[h >= (1 << log2c) - 64]
    keys = np.concatenate([tail[:300], cand[h < 8][:10], cand[(h > 500) & (h < 900)][:300]])
    vals = np.arange(1, keys.size + 1, dtype=np.uint64)
    t, o = cuda_lib.Table(1 << log2c), oracle_mod.OracleTable(1 << log2c)
    t.build(to_dev(keys), to_dev(vals))
    assert o.build(keys, vals) == 0
    assert _cells(t)[0, 0] != 0
    bk = np.concatenate([tail[290:400], cand[h < 8][5:20]])
    t.merge(to_dev(bk), to_dev(bk))
    assert o.merge(bk, bk) == 0
    assert np.array_equal(_cells(t), o.cells())


@pytest.mark.parametrize("n,distinct", [(4095, 4095), (4096, 3000), (4097, 4097), (1_300_001, 1_000_000),
                                        (1_300_001, 7)])
def test_build_at_tile_edges(cuda_lib, oracle_mod, n, distinct):
    # 4096 cells a tile; 1.3 M cells are more tiles than run at once
    rng = np.random.default_rng(n)
    base = W.uniform_keys(distinct, start=n, seed=73)
    keys = base if n == distinct else base[rng.integers(0, distinct, n)]
    vals = rng.integers(1, 1 << 62, n).astype(np.uint64)
    c = 1 << int(np.ceil(np.log2(n / 0.75)))
    t, o = cuda_lib.Table(c), oracle_mod.OracleTable(c)
    t.build(to_dev(keys), to_dev(vals))
    assert o.build(keys, vals) == 0
    assert np.array_equal(_cells(t), o.cells())
    assert t.size() == (o.live, o.nonempty, c)
