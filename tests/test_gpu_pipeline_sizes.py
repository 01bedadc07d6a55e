"""Pinned host arrays of a few operations more than a multiple of eight pieces:
every piece has its own copies and events.  Equal to the same calls on device
arrays.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(1 << 20) + 1, (1 << 20) + 7, (1 << 22) + 3])
def test_ragged_sizes(cuda_lib, n):
    import torch

    keys = W.uniform_keys(n, seed=93)
    q = W.uniform_keys(n, start=n // 2, seed=93)
    pin = lambda a: torch.from_numpy(a.view(np.int64)).pin_memory()  # noqa: E731
    got = []
    for put in (pin, to_dev):
        arrays = [put(keys), put(keys * np.uint64(3)), put(q)]
        out = [torch.full((n,), 9, dtype=d) for d in (torch.uint8, torch.uint8, torch.int64, torch.uint8)]
        out = [x.pin_memory() if put is pin else x.cuda() for x in out]
        t = cuda_lib.Table(1 << 24)
        t.insert(arrays[0], arrays[1], out[0])
        t.find(arrays[2], out[2], out[1])
        t.erase(arrays[2], out[3])
        torch.cuda.synchronize()
        got.append([x.cpu().numpy() for x in out] + [np.array(t.size(check=True))])
    for x, y in zip(*got):
        assert np.array_equal(x, y)
