"""Pinned calls on different streams: each waits for its own stream's work
alone, and more of them than copy lanes exist give the same results.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

N = (1 << 20) + 5


def _setup(cuda_lib, i):
    import torch

    keys = W.uniform_keys(N, start=i * N, seed=95)
    t = cuda_lib.Table(1 << 22)
    t.insert(to_dev(keys), to_dev(keys * np.uint64(i + 3)))
    pin = torch.from_numpy(keys.view(np.int64)).pin_memory()
    return t, keys * np.uint64(i + 3), pin, torch.zeros(N, dtype=torch.int64).pin_memory()


def test_a_busy_stream_does_not_hold_up_another(cuda_lib):
    import torch

    (ta, wa, ka, oa), (tb, wb, kb, ob) = _setup(cuda_lib, 0), _setup(cuda_lib, 1)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for t, k, o, s in ((ta, ka, oa, a), (tb, kb, ob, b)):  # first calls: streams and events are made
        t.find(k, o, stream=s)
    torch.cuda.synchronize()
    oa.zero_(), ob.zero_()
    with torch.cuda.stream(a):
        torch.cuda._sleep(600_000_000)  # about 0.3 s
    busy = torch.cuda.Event()
    busy.record(a)
    ta.find(ka, oa, stream=a)
    tb.find(kb, ob, stream=b)
    b.synchronize()
    assert not busy.query()  # b is done, a has not begun
    assert np.array_equal(ob.numpy().view(np.uint64), wb)
    a.synchronize()
    assert np.array_equal(oa.numpy().view(np.uint64), wa)


def test_more_streams_than_lanes(cuda_lib):
    import torch

    every = [_setup(cuda_lib, i) for i in range(7)]
    streams = [torch.cuda.Stream() for _ in every]
    torch.cuda.synchronize()
    for _ in range(3):
        for (t, _, k, o), s in zip(every, streams):
            o.zero_()
            with torch.cuda.stream(s):
                torch.cuda._sleep(2_000_000)
            t.find(k, o, stream=s)
        for (_, want, _, o), s in zip(every, streams):
            s.synchronize()
            assert np.array_equal(o.numpy().view(np.uint64), want)
    for (t, *_), s in zip(every, streams):
        s.synchronize()
        t.destroy()
