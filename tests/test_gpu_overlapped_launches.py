"""Calls issued back to back on one stream, whose launches overlap: every call
sees what the ones before it wrote.  Tables small enough that several launches
fit the GPU at once, contents that change from call to call (so that a stale
read shows), no synchronisation until the end.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import to_dev, to_np_u8, to_np_u64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2c,n", [(8, 60), (11, 900), (14, 7000), (18, 100_000)])
@pytest.mark.parametrize("width", [0, -1, 1, 4])
def test_changing_contents(cuda_lib, log2c, n, width):
    import torch

    rounds = 24
    keys = W.uniform_keys(3 * n, start=log2c * 10**6, seed=121)
    k = [to_dev(keys[i * n:(i + 1) * n]) for i in range(3)]
    vals = [[to_dev(keys[i * n:(i + 1) * n] * np.uint64(r + 3)) for i in range(2)] for r in range(rounds)]
    probe = to_dev(np.concatenate([keys[:2 * n:2], keys[2 * n:]]))
    m = probe.numel()
    outs = torch.full((rounds, 4, m), -7, dtype=torch.int64, device="cuda")
    found = torch.full((rounds, 4, m), 9, dtype=torch.uint8, device="cuda")
    t = cuda_lib.Table(1 << log2c)
    t.set_config(group_width=width)
    torch.cuda.synchronize()
    for r in range(rounds):
        t.clear()
        t.find(probe, outs[r, 0], found[r, 0])
        t.insert(k[r % 2], vals[r][r % 2])
        t.find(probe, outs[r, 1], found[r, 1])
        t.insert_or_update(k[r % 2], vals[r][(r + 1) % 2], cuda_lib.OVERWRITE)
        t.find(probe, outs[r, 2], found[r, 2])
        if r % 4 == 3:
            t.migrate(2 << log2c)
        t.erase(k[r % 2])
        t.find(probe, outs[r, 3], found[r, 3])
        if r % 4 == 3:
            t.migrate(1 << log2c)  # (shrinking waits for the count; the other rounds run on without)
    torch.cuda.synchronize()
    o, f = to_np_u64(outs).reshape(rounds, 4, m), to_np_u8(found).reshape(rounds, 4, m)
    p = to_np_u64(probe)
    at = np.concatenate([np.arange(0, 2 * n, 2), np.arange(2 * n, 3 * n)])  # probe = keys[at]
    for r in range(rounds):
        i = r % 2
        mine = at // n == i
        first = p * np.uint64(r + 3)
        second = keys[np.where(mine, (1 - i) * n + at % n, 0)] * np.uint64(r + 3)
        for call, present, want in ((0, mine & False, first), (1, mine, first), (2, mine, second), (3, mine & False, first)):
            assert np.array_equal(f[r, call], present.astype(np.uint8)), (r, call)
            assert np.array_equal(o[r, call], np.where(present, want, np.uint64(0))), (r, call)


@pytest.mark.parametrize("n", [50, 3000, 40_000])
def test_builds_and_merges_in_turn(cuda_lib, n):
    import torch

    rounds = 16
    t = cuda_lib.Table(max(64, 4 << int(np.ceil(np.log2(n)))))
    ks = [W.uniform_keys(n, start=r * n, seed=122) for r in range(rounds + 1)]
    dk = [to_dev(x) for x in ks]
    dv = [to_dev(x * np.uint64(5)) for x in ks]
    q = to_dev(np.concatenate(ks))
    out = torch.full((rounds, 2, q.numel()), -7, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for r in range(rounds):
        t.clear()
        t.build(dk[r], dv[r])
        t.find(q, out[r, 0])
        t.merge(dk[r + 1][: n // 2], dv[r + 1][: n // 2])
        t.find(q, out[r, 1])
    torch.cuda.synchronize()
    o = to_np_u64(out).reshape(rounds, 2, rounds + 1, n)
    for r in range(rounds):
        want = np.zeros((rounds + 1, n), np.uint64)
        want[r] = ks[r] * np.uint64(5)
        assert np.array_equal(o[r, 0], want), r
        want[r + 1, : n // 2] = ks[r + 1][: n // 2] * np.uint64(5)
        assert np.array_equal(o[r, 1], want), r
