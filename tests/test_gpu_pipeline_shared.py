"""Pinned result arrays that share memory with the keys: the inputs are read
before any result is written, whatever the shift between them.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1, 1 << 17, (1 << 20) + 3, -1, -(1 << 17)])
def test_results_over_keys(cuda_lib, shift):
    import torch

    n = (1 << 20) + 9
    keys = W.uniform_keys(n, seed=95)
    t = cuda_lib.Table(1 << 22)
    t.insert(to_dev(keys), to_dev(keys * np.uint64(3)))
    memory = torch.zeros(n + abs(shift), dtype=torch.int64).pin_memory()
    q, out = memory[max(-shift, 0):][:n], memory[max(shift, 0):][:n]
    codes = torch.full((n,), 9, dtype=torch.uint8).pin_memory()
    q.copy_(torch.from_numpy(keys.view(np.int64)))
    t.find(q, out, codes)
    torch.cuda.synchronize()
    assert np.array_equal(out.numpy().view(np.uint64), keys * np.uint64(3))
    assert bool((codes == 1).all())


def test_codes_over_keys(cuda_lib):
    import torch

    n = (1 << 20) + 9
    keys = W.uniform_keys(n, seed=96)
    t = cuda_lib.Table(1 << 22)
    memory = torch.from_numpy(keys.view(np.int64).copy()).pin_memory()
    codes = memory.view(torch.uint8)[5 << 20:][:n]  # over keys of a later piece
    t.insert(memory, to_dev(keys * np.uint64(3)), codes)
    torch.cuda.synchronize()
    assert bool((codes == 1).all())
    assert t.size(check=True)[0] == n
    out = torch.zeros(n, dtype=torch.int64, device="cuda")
    t.find(to_dev(keys), out)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), keys * np.uint64(3))
