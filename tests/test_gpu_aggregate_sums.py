"""insertOrUpdate and update folded in shared memory: sums of full 64-bit values
(kept as two 32-bit words with a carry) modulo 2^64, overwrites, and codes, at
the edges of the 1024-operation window and with few, many and all-equal keys.
Expected sums come from numpy's uint64 arithmetic: equality, no tolerance.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import codes_buf, to_dev, to_np_u8, to_np_u64, vals_buf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,distinct", [(1, 1), (1023, 1), (1024, 1024), (1025, 3), (70_001, 1), (70_001, 40),
                                        (300_000, 60_000), (1_000_003, 900_000)])
@pytest.mark.parametrize("agg,load", [(1, 0.4), (1, 0.9), (2, 0.4), (3, 0.4)])
def test_folded_sums_and_codes(cuda_lib, n, distinct, agg, load):
    rng = np.random.default_rng(n + distinct)
    base = W.uniform_keys(distinct, start=n, seed=101)
    pick = rng.integers(0, distinct, n)
    pick[:min(n, distinct)] = np.arange(min(n, distinct))
    pick = rng.permutation(pick)
    used = np.unique(pick)
    # values around and above 2^32, and ones whose sums wrap past 2^64
    vals = rng.integers(0, 1 << 63, n, dtype=np.uint64) * np.uint64(2) + rng.integers(0, 2, n, dtype=np.uint64)
    vals[::3] = (1 << 32) - 1
    vals[1::7] = 1
    keys = base[pick]
    want = np.zeros(distinct, np.uint64)
    np.add.at(want, pick, vals)

    cap = max(64, 1 << int(np.ceil(np.log2(distinct / load))))
    t = cuda_lib.Table(cap)
    t.set_config(iou_aggregate=agg)
    codes = codes_buf(n)
    t.insert_or_update(to_dev(keys), to_dev(vals), cuda_lib.ADD, codes)
    c = to_np_u8(codes)
    assert c.max() <= 1
    first = np.bincount(pick, weights=c, minlength=distinct)
    assert (first[used] == 1).all()  # one operation per key inserted it
    got = vals_buf(used.size)
    t.find(to_dev(base[used]), got)
    assert np.array_equal(to_np_u64(got), want[used])
    # update the same keys, mixed with absent ones, then overwrite
    absent = W.uniform_keys(n, start=10**8, seed=101)
    q = np.where(rng.random(n) < 0.7, keys, absent)
    codes = codes_buf(n)
    t.update(to_dev(q), to_dev(vals), cuda_lib.ADD, codes)
    assert np.array_equal(to_np_u8(codes), (q == keys).astype(np.uint8))
    np.add.at(want, pick[q == keys], vals[q == keys])
    t.find(to_dev(base[used]), got)
    assert np.array_equal(to_np_u64(got), want[used])
    t.insert_or_update(to_dev(keys), to_dev(keys * np.uint64(7)), cuda_lib.OVERWRITE, codes)
    assert (to_np_u8(codes) == 0).all()
    t.find(to_dev(base[used]), got)
    assert np.array_equal(to_np_u64(got), base[used] * np.uint64(7))
    assert t.size(check=True) == (used.size, used.size, cap)
