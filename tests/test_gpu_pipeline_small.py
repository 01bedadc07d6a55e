"""Pinned host arrays of 2^20 to 2^24 operations: staged whole, copied and run
in pieces of an eighth.  Sizes lie at the limits of that range and give a last
piece of one operation.  Results equal the same calls on device arrays (whole
numbers, one right answer each), with any subset of the arrays on the host.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

LO = 1 << 20


@pytest.mark.parametrize("n", [LO - 1, LO, 7 * (3 << 16) + 1, (1 << 24)])
@pytest.mark.parametrize("growable,mixed", [(False, False), (True, False), (False, True)])
def test_pieces_match_device_arrays(cuda_lib, n, growable, mixed):
    import torch

    keys = W.uniform_keys(n, seed=91)
    q = np.concatenate([keys[::2], W.uniform_keys(n - keys[::2].size, start=10**9, seed=91)])
    got, keep = [], []  # the arrays of a call stay alive until it is done
    for host in (True, False):
        def arr(a, on_host=True):
            t = torch.from_numpy(np.ascontiguousarray(a).view(np.int64))
            keep.append(t.pin_memory() if host and on_host else t.cuda())
            return keep[-1]

        def out(dtype, on_host=True):
            t = torch.full((n,), 9, dtype=dtype)
            return t.pin_memory() if host and on_host else t.cuda()

        t = cuda_lib.Table(1 << 12 if growable else 1 << 26, growable=growable)
        ci, cu, ce, fo, vo = [out(torch.uint8) for _ in range(4)] + [out(torch.int64, not mixed)]
        t.insert(arr(keys), arr(keys * np.uint64(3), not mixed), ci)
        t.find(arr(q), vo, fo)
        t.update(arr(q, not mixed), arr(keys), cuda_lib.ADD, cu)
        t.insert_or_update(arr(q), arr(keys), cuda_lib.OVERWRITE)
        t.erase(arr(keys), ce)
        torch.cuda.synchronize()
        sums = torch.zeros(n, dtype=torch.int64, device="cuda")
        t.find(to_dev(q), sums)
        got.append([x.cpu().numpy() for x in (ci, fo, vo, cu, ce, sums)] + [np.array(t.size(check=True))])
    for x, y in zip(*got):
        assert np.array_equal(x, y)
