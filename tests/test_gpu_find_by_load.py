"""Large finds on a table whose non-empty cells the host only bounds: several
launches are made, each for a band of loads, and the one for the table's
actual load answers.  Loads on both sides of every band edge, with the bound
far above them (most of the inserted batch repeats a few keys).  Results are
whole numbers known from the inputs.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import codes_buf, to_dev, to_np_u8, to_np_u64, vals_buf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2c", [20, 23, 25])
@pytest.mark.parametrize("load", [0.01, 0.3749, 0.3751, 0.599, 0.601, 0.799, 0.85])
def test_answers_at_any_load(cuda_lib, log2c, load):
    c = 1 << log2c
    live = int(c * load)
    keys = W.uniform_keys(live, start=log2c, seed=111)
    t = cuda_lib.Table(c)
    t.insert(to_dev(keys), to_dev(keys * np.uint64(3)))
    again = np.repeat(keys[:16], c // 16)
    t.insert(to_dev(again), to_dev(again))  # nothing new, but the bound passes c
    n = (1 << 22) + 77
    rng = np.random.default_rng(live)
    present = rng.random(n) < 0.5
    q = np.where(present, keys[rng.integers(0, live, n)], W.uniform_keys(n, start=10**9, seed=111))
    out, codes = vals_buf(n), codes_buf(n)
    t.find(to_dev(q), out, codes)
    assert np.array_equal(to_np_u64(out), np.where(present, q * np.uint64(3), np.uint64(0)))
    assert np.array_equal(to_np_u8(codes), present.astype(np.uint8))
