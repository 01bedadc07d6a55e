"""Finds on tables on both sides of the size up to which results are stored
directly (2^25 cells) rather than through the warp's ring, for the two windows
that have both forms.  Results are whole numbers known from the inputs:
equality, no tolerance.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import codes_buf, to_dev, to_np_u8, to_np_u64, vals_buf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v", [4])
@pytest.mark.parametrize("g", [1, 2])
@pytest.mark.parametrize("log2c,live", [(8, 200), (24, 1 << 16), (25, 1 << 16), (26, 1 << 16)])
@pytest.mark.parametrize("n", [1, 255, 50_001])
def test_find_forms(cuda_lib, g, v, log2c, live, n):
    keys = W.uniform_keys(live, start=3_000_000, seed=67)
    t = cuda_lib.Table(1 << log2c)
    t.insert(to_dev(keys), to_dev(keys * np.uint64(3)))
    t.set_config(group_width=g, lane_cells=v)
    rng = np.random.default_rng(n)
    present = rng.random(n) < 0.5
    q = np.where(present, keys[rng.integers(0, live, n)], W.uniform_keys(n, start=9_000_000, seed=67))
    out, codes = vals_buf(n + 8), codes_buf(n)
    t.find(to_dev(q), out, codes)
    got = to_np_u64(out)
    assert np.array_equal(got[:n], np.where(present, q * np.uint64(3), np.uint64(0)))
    assert np.array_equal(got[n:], to_np_u64(vals_buf(n + 8))[n:])
    assert np.array_equal(to_np_u8(codes), present.astype(np.uint8))
