"""Large finds on a table whose non-empty cells the host only bounds: both
sides of the last band's edge, and every band of the largest table sizes.
Results are whole numbers known from the inputs.
"""
import pytest

import workloads as W
from gpu_helpers import codes_buf, vals_buf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2c,load", [(c, x) for c in (20, 23, 25) for x in (0.874, 0.876, 0.95)]
                         + [(27, x) for x in (0.3, 0.5, 0.7, 0.85, 0.9)])
def test_answers_at_any_load(cuda_lib, log2c, load):
    import torch

    c = 1 << log2c
    live, n = int(c * load), (1 << 22) + 77
    every = W.uniform_keys(live + n, start=log2c, seed=111, backend="cuda")
    keys = every[:live]
    t = cuda_lib.Table(c)
    t.insert(keys, keys * 3)
    again = keys[:16].repeat(c // 16)
    t.insert(again, again)  # nothing new, but the bound passes c
    gen = torch.Generator(device="cuda").manual_seed(live)
    present = torch.rand(n, device="cuda", generator=gen) < 0.5
    at = torch.randint(0, live, (n,), device="cuda", generator=gen)
    q = torch.where(present, keys[at], every[live:])
    out, codes = vals_buf(n), codes_buf(n)
    t.find(q, out, codes)
    assert torch.equal(out, torch.where(present, q * 3, 0))
    assert torch.equal(codes, present.to(torch.uint8))
