"""Finds on a table of 2^26 cells, the smallest whose one-line windows keep
their results in the warp's ring: one CTA per SM makes each warp's slice several
hundred operations long, so the ring wraps, and the keys' homes lie in a narrow
range of cells filled to 0.97, so some probes outlast the window that their
result belongs to.  Results are whole numbers known from the inputs: equality,
no tolerance.
"""
import numpy as np
import pytest

from gpu_helpers import codes_buf, to_dev, to_np_u8, to_np_u64, vals_buf

pytestmark = pytest.mark.gpu

LOG2C, REGION = 26, 1 << 18  # the region: cells that the keys are homed in


def _unmix(h):
    """The key whose fmix64 is h: both multipliers are odd (inverses modulo
    2^64), and x ^= x >> 33 undoes itself."""
    for m in (0xC4CEB9FE1A85EC53, 0xFF51AFD7ED558CCD):
        h = h ^ (h >> np.uint64(33))
        h = h * np.uint64(pow(m, -1, 1 << 64))
    return h ^ (h >> np.uint64(33))


@pytest.mark.parametrize("g", [1, 2])
@pytest.mark.parametrize("per_warp,with_codes", [(64, True), (129, False), (700, True)])
def test_slices_many_windows_long(cuda_lib, g, per_warp, with_codes):
    import torch

    rng = np.random.default_rng(per_warp)
    live = int(REGION * 0.97)
    n = torch.cuda.get_device_properties(0).multi_processor_count * 8 * per_warp - 5
    # distinct hashes of the region: any cell of it, a counter in the low bits
    cell = rng.integers(0, REGION, live + n, dtype=np.uint64) + np.uint64(12345)
    keys = _unmix((cell << np.uint64(64 - LOG2C)) | np.arange(live + n, dtype=np.uint64))
    held, absent = keys[:live], keys[live:]
    t = cuda_lib.Table(1 << LOG2C)
    t.insert(to_dev(held), to_dev(held * np.uint64(3)))
    t.set_config(group_width=g, lane_cells=4, ctas_per_sm=1)
    present = rng.random(n) < 0.5
    q = np.where(present, held[rng.integers(0, live, n)], absent)
    out, codes = vals_buf(n + 8), codes_buf(n + 8)
    t.find(to_dev(q), out, codes if with_codes else None)
    got = to_np_u64(out)
    assert np.array_equal(got[:n], np.where(present, q * np.uint64(3), np.uint64(0)))
    assert np.array_equal(got[n:], to_np_u64(vals_buf(8)))
    if with_codes:
        assert np.array_equal(to_np_u8(codes)[:n], present.astype(np.uint8))
