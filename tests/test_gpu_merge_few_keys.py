"""Bulk merges whose batches leave long ranges of empty cells: copies of few
keys, keys of one part of the hash range.  The cells equal the oracle's bit for
bit, and the time stays near that of a batch of as many distinct keys (which
moves more): one CTA writing the empty cells alone took ten times as long.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import to_dev, to_np_u64

pytestmark = pytest.mark.gpu

LOG2C = 20


def _batch(kind, n, homes):
    pool = W.uniform_keys(12 * n, seed=131)
    h = homes(pool, LOG2C)
    c = 1 << LOG2C
    if kind == "low":  # the first eighth of the table
        return pool[h < c // 8][:n]
    if kind == "high":  # the last: the tail wraps to the first cells
        return np.concatenate([pool[h >= c - c // 8][:n - 64], np.repeat(pool[h >= c - 4][:4], 16)])
    if kind == "edges":  # gaps of 2^16 - 1, 2^16 and 2^16 + 1 cells and a full part
        at = np.cumsum([0, 1 << 16, (1 << 16) + 1, (1 << 16) + 2])
        return np.concatenate([[pool[h >= x][np.argmin(h[h >= x])] for x in at], pool[h >= 3 * c // 4][:n]])
    return np.repeat(pool[:kind], -(-n // kind))[:n]


@pytest.mark.parametrize("kind", [1, 3, 40, "low", "high", "edges"])
@pytest.mark.parametrize("before", [0, 5, 1000])
def test_long_ranges(cuda_lib, oracle_mod, kind, before):
    n = 1 << 17  # an eighth of the cells
    keys = _batch(kind, n, oracle_mod.homes)
    vals = np.arange(1, keys.size + 1, dtype=np.uint64)
    t, o = cuda_lib.Table(1 << LOG2C), oracle_mod.OracleTable(1 << LOG2C)
    if before:
        b = W.uniform_keys(before, start=10**9, seed=131)
        t.build(to_dev(b), to_dev(b))
        o.build(b, b)
    t.merge(to_dev(keys), to_dev(vals))
    assert o.merge(keys, vals) == 0
    assert np.array_equal(to_np_u64(t.cells()).reshape(-1, 2), o.cells())
    assert t.size(check=True) == (o.live, o.nonempty, o.capacity)


def test_time_of_copies(cuda_lib):
    import torch

    n = 1 << 24
    distinct = to_dev(W.uniform_keys(n, seed=132))
    copies = distinct[:16].repeat(n // 16)
    took = {}
    for name, k in (("copies", copies), ("distinct", distinct)):
        for _ in range(4):
            t = cuda_lib.Table(2 * n)
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            t.merge(k, k)
            b.record()
            torch.cuda.synchronize()
            took[name] = min(took.get(name, 1e9), a.elapsed_time(b))
            t.destroy()
    assert took["copies"] < 2 * took["distinct"], took
