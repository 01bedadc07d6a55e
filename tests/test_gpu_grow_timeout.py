"""In-kernel growth whose bounded wait runs out while a migration is under way:
the table stays valid, and the next migration counts from zero.

One cluster of 2^15 cells (keys homed at consecutive cells, so that filling it
probes nothing) is one lane's work for several milliseconds, which the other
blocks wait for with a limit of 300 us; the table stands at its threshold, so
the launch migrates before it inserts anything.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import to_dev, to_np_u64

pytestmark = pytest.mark.gpu


def _keys_homed_at(homes, log2c):
    """Keys whose hash (the 64-bit finalizer of MurmurHash3) has these top bits."""
    x = (homes.astype(np.uint64) << np.uint64(64 - log2c)) | np.uint64(0x1234567)
    for c in (0xc4ceb9fe1a85ec53, 0xff51afd7ed558ccd):
        x ^= x >> np.uint64(33)
        x *= np.uint64(pow(c, -1, 1 << 64))
    return x ^ (x >> np.uint64(33))


def test_wait_runs_out_in_a_migration(cuda_lib, oracle_mod):
    log2c, n = 16, 1 << 15
    keys = _keys_homed_at(np.arange(n), log2c)
    assert np.array_equal(oracle_mod.homes(keys, log2c), np.arange(n))
    t = cuda_lib.Table(1 << log2c, growable=True)
    t.insert(to_dev(keys), to_dev(keys * np.uint64(3)))
    assert t.size() == (n, n, 1 << log2c)
    more = W.uniform_keys(1000, seed=85)
    t.set_config(grow_in_kernel=1, grow_spin_us=300)
    with pytest.raises(cuda_lib.ChtError) as ei:
        t.insert(to_dev(more), to_dev(more))
    assert ei.value.status == cuda_lib.CHT_ERR_TIMEOUT
    assert t.size(check=True) == (n, n, 1 << log2c)  # nothing was inserted, the migration was dropped
    t.set_config(grow_in_kernel=0, grow_spin_us=0)
    t.migrate(2 << log2c)
    assert t.size(check=True) == (n, n, 2 << log2c)
    t.merge(to_dev(more), to_dev(more))
    assert t.size(check=True)[:2] == (n + more.size, n + more.size)
    ek, ev = map(to_np_u64, t.export())
    want = {**dict(zip(keys.tolist(), (keys * np.uint64(3)).tolist())), **dict(zip(more.tolist(), more.tolist()))}
    assert dict(zip(ek.tolist(), ev.tolist())) == want and ek.size == len(want)
