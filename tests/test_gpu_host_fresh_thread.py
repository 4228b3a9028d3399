"""A page-locked array is read in place whatever the calling thread did before:
a thread's first CUDA call, on a stream that another thread has used, allocates
no staging buffers (128 MiB of device memory)."""
import ctypes
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_first_call_of_a_thread_is_in_place(sr):
    n = 1 << 16
    big = torch.arange(3 * n, dtype=torch.int32).pin_memory()  # the array lies inside an allocation
    warm, out = ctypes.c_int64(-1), ctypes.c_int64(-1)
    s1 = torch.cuda.Stream()
    sr.check(sr.reduce_sum_host_ptr(big.data_ptr() + 4 * n, n, sr.I32, ctypes.addressof(warm), None, s1.cuda_stream))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    status = []
    t = threading.Thread(target=lambda: status.append(sr.reduce_sum_host_ptr(
        big.data_ptr() + 4 * n, n, sr.I32, ctypes.addressof(out), None, s1.cuda_stream)))
    t.start()
    t.join()
    assert status == [sr.OK]
    assert out.value == warm.value == int(big[n:2 * n].sum())
    assert before - torch.cuda.mem_get_info()[0] < 64 << 20
