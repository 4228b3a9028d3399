"""sr_reduce_sum_host around the size up to which page-locked arrays are read in
place: every dtype, a start off the vector alignment, an array inside a larger
page-locked one; integer values, so every path gives the exact sum."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu
LIMIT = 128 << 20  # bytes


@pytest.mark.parametrize("dtype_name", ["F32", "I32", "BF16", "FP8E4M3"])
def test_in_place_limit(sr, dtype_name):
    dt = getattr(sr, dtype_name)
    eb = {sr.F32: 4, sr.I32: 4, sr.BF16: 2, sr.FP8E4M3: 1}[dt]
    n_max = LIMIT // eb + 8
    v = workloads.uniform_i32(n_max, seed=5, lo=-4, hi=4)
    t = torch.from_numpy(v)
    t = {sr.F32: lambda: t.float(), sr.I32: lambda: t, sr.BF16: lambda: t.bfloat16(),
         sr.FP8E4M3: lambda: t.float().to(torch.float8_e4m3fn).view(torch.uint8)}[dt]()
    pinned = t.pin_memory()
    out = np.zeros(1, np.int64 if dt == sr.I32 else np.float32)
    for n in (1, 3, 1000, LIMIT // eb - 1, LIMIT // eb, LIMIT // eb + 1):
        for off in (0, 1, 5):
            for stage in (sr.AUTO, sr.TWO_KERNEL):
                out[0] = -1
                sr.check(sr.reduce_sum_host_ptr(pinned.data_ptr() + off * eb, n, dt, out.ctypes.data,
                                                sr.make_config(stage)))
                want = oracle.sum_i32(np.ascontiguousarray(v[off:off + n]))
                assert out[0] == want, (dtype_name, n, off, stage)
    assert sr.stream_release() == sr.OK  # frees the result slots too; the next call makes them again
    sr.check(sr.reduce_sum_host_ptr(pinned.data_ptr(), 100, dt, out.ctypes.data, None))
    assert out[0] == int(v[:100].sum())
