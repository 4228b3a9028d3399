"""More host threads blocked in sr_reduce_sum_host on one stream than the library
has result slots: every thread gets its own array's sum."""
import ctypes
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant_name", ["AUTO", "F_HOST_DIRECT", "TWO_KERNEL"])  # the last by copies
def test_two_hundred_threads_on_one_stream(sr, variant_name):
    threads, n = 200, 1 << 12
    stream = torch.cuda.Stream()
    x = torch.ones(threads, n, dtype=torch.int32).mul_(torch.arange(threads, dtype=torch.int32)[:, None]).pin_memory()
    cfg = sr.make_config(getattr(sr, variant_name))
    warm = ctypes.c_int64(-1)
    sr.check(sr.reduce_sum_host_ptr(x[1].data_ptr(), n, sr.I32, ctypes.addressof(warm), cfg, stream.cuda_stream))
    assert warm.value == n
    got = [ctypes.c_int64(-1) for _ in range(threads)]
    status = [None] * threads

    def call(k):
        status[k] = sr.reduce_sum_host_ptr(x[k].data_ptr(), n, sr.I32, ctypes.addressof(got[k]), cfg,
                                           stream.cuda_stream)

    with torch.cuda.stream(stream):
        torch.cuda._sleep(400_000_000)  # 0.2 s: all calls are queued before the first runs
    ts = [threading.Thread(target=call, args=(k,)) for k in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert status == [sr.OK] * threads
    assert [g.value for g in got] == [k * n for k in range(threads)]
