"""Finds whose warps run many operations each, with results kept in the warp's
ring and written 32 at a time (one-line probe windows).

One CTA per SM makes each warp's slice of the batch a few windows long, so the
ring wraps, and at load 0.97 some probes outlast the window their result
belongs to and store it themselves.  Slice lengths cover less than a window,
whole windows, one more than the ring, and many times the ring.  Results are
whole numbers known from the inputs: equality, no tolerance.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import codes_buf, to_dev, to_np_u8, to_np_u64, vals_buf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g,v", [(1, 2), (2, 2), (2, 4), (4, 2), (8, 1), (4, 4)])
@pytest.mark.parametrize("load,per_warp,with_codes", [(0.5, 31, True), (0.97, 64, True), (0.97, 129, False),
                                                      (0.97, 700, True)])
def test_find_results_by_window(cuda_lib, g, v, load, per_warp, with_codes):
    import torch

    log2c = 18
    live = int((1 << log2c) * load)
    keys = W.uniform_keys(live, start=3_000_000, seed=61)
    t = cuda_lib.Table(1 << log2c)
    t.insert(to_dev(keys), to_dev(keys * np.uint64(3)))
    t.set_config(group_width=g, lane_cells=v, ctas_per_sm=1)
    n = torch.cuda.get_device_properties(0).multi_processor_count * 8 * per_warp - 5
    rng = np.random.default_rng(per_warp)
    present = rng.random(n) < 0.5
    q = np.where(present, keys[rng.integers(0, live, n)], W.uniform_keys(n, start=9_000_000, seed=61))
    none = rng.integers(0, n, 20)
    q[none], present[none] = 0, False  # a reserved key: code 3, value 0
    out, codes = vals_buf(n + 8), codes_buf(n + 8)
    t.find(to_dev(q), out, codes if with_codes else None)
    got = to_np_u64(out)
    assert np.array_equal(got[:n], np.where(present, q * np.uint64(3), np.uint64(0)))
    untouched = to_np_u64(vals_buf(n + 8))[n:]
    assert np.array_equal(got[n:], untouched)
    if with_codes:
        assert np.array_equal(to_np_u8(codes)[:n], np.where(q == 0, 3, present).astype(np.uint8))
