"""The bulk build's sort at the edges of its tiles.  The layout is deterministic: cells equal the oracle's bit for bit.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import to_dev, to_np_u64

pytestmark = pytest.mark.gpu

def _cells(t):
    return to_np_u64(t.cells()).reshape(-1, 2)


@pytest.mark.parametrize("n,distinct", [(4095, 4095), (4096, 3000), (4097, 4097), (1_300_001, 1_000_000),
                                        (1_300_001, 7)])
def test_build_at_tile_edges(cuda_lib, oracle_mod, n, distinct):
    # 4096 cells a tile; 1.3 M cells are more tiles than run at once
    rng = np.random.default_rng(n)
    base = W.uniform_keys(distinct, start=n, seed=73)
    keys = base if n == distinct else base[rng.integers(0, distinct, n)]
    vals = rng.integers(1, 1 << 62, n).astype(np.uint64)
    c = 1 << int(np.ceil(np.log2(n / 0.75)))
    t, o = cuda_lib.Table(c), oracle_mod.OracleTable(c)
    t.build(to_dev(keys), to_dev(vals))
    assert o.build(keys, vals) == 0
    assert np.array_equal(_cells(t), o.cells())
    assert t.size() == (o.live, o.nonempty, c)
