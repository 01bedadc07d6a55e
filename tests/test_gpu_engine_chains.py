"""Engine launches bound by one table's chain of levels: the items of a group
are loaded ahead of the item before them.  One table has a long chain (which
makes the launch take that way), one a large batch (so that the launch's work
exceeds the short chains and their items keep up to 256 operations), and one a
group of dependent batches of the size under test.  Results equal the same
batches as single calls; all are whole numbers with one right answer.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import codes_buf, to_dev, to_np_u8, to_np_u64, vals_buf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [1, 31, 32, 33, 200, 256])
@pytest.mark.parametrize("reuse", [0, 1])
def test_group_items_loaded_ahead(cuda_lib, size, reuse):
    cht = cuda_lib
    big = W.uniform_keys(1_000_000, start=0, seed=81)
    keys = W.uniform_keys(4096, start=5_000_000, seed=81)

    def ops(tables):
        a, b, c = tables
        out = [(c, cht.OP_INSERT, big, big, False)]
        for r in range(30):  # the long chain
            k = keys[r * 64:(r + 1) * 64]
            out.append((a, cht.OP_INSERT, k, k * np.uint64(5), False))
            out.append((a, cht.OP_FIND, k, None, True))
        k = keys[:size]
        out += [(b, cht.OP_INSERT, k, k * np.uint64(3), False), (b, cht.OP_FIND, k, None, True),
                (b, cht.OP_UPDATE_ADD, k, k, False), (b, cht.OP_ERASE, k[: (size + 1) // 2], None, False),
                (b, cht.OP_FIND, k, None, True), (b, cht.OP_INSERT, k, k, False), (b, cht.OP_FIND, k, None, True)]
        return out

    def make():
        ts = [cht.Table(1 << 13), cht.Table(1 << 11), cht.Table(1 << 21)]
        for t in ts:
            t.set_config(reuse_tombstones=reuse)
        return ts

    results = []
    for planned in (True, False):
        tables, entries = make(), []
        for t, op, k, v, find in ops(tables):
            entries.append((t, op, to_dev(k), None if v is None else to_dev(v), vals_buf(k.size) if find else None,
                            codes_buf(k.size)))
        if planned:
            plan = cht.Plan(entries)
            plan.launch()
            assert plan.status() == 0
        else:
            for t, op, k, v, vo, co in entries:
                if op == cht.OP_INSERT:
                    t.insert(k, v, co)
                elif op == cht.OP_FIND:
                    t.find(k, vo, co)
                elif op == cht.OP_UPDATE_ADD:
                    t.update(k, v, cht.ADD, co)
                else:
                    t.erase(k, co)
        results.append([(to_np_u8(co), None if vo is None else to_np_u64(vo)) for _, _, _, _, vo, co in entries] +
                       [t.size() for t in tables])
    for x, y in zip(*results):
        if isinstance(x[0], np.ndarray):
            assert np.array_equal(x[0], y[0])
            assert (x[1] is None) == (y[1] is None) and (x[1] is None or np.array_equal(x[1], y[1]))
        else:
            assert x == y
