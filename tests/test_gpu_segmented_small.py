"""Small segmented calls: the strip kernel's smallest piece (a whole chunk from a
mean of 160 bytes per segment, a quarter below) either side of the line, in
every finish, results exact; and the default form's time against the LDG
kernel's on the same call, where the pieces decide it."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,eb", [(torch.int32, 4), (torch.float32, 4), (torch.bfloat16, 2), (torch.uint8, 1)])
def test_either_side_of_the_mean(sr, dtype, eb):
    for nseg in (1, 7, 300, 5000):
        for total in (160 * nseg // eb - 1, 160 * nseg // eb, 160 * nseg // eb + 1, 30 * nseg,
                      3648 * 3072 // eb - 5, 3648 * 3072 // eb + 3000):  # three quarters of a chunk to a warp
            rng = np.random.default_rng(total)
            cuts = np.sort(rng.integers(0, total + 1, nseg - 1))
            off = np.concatenate([[0], cuts, [total]]).astype(np.int64)
            if dtype == torch.uint8:  # E4M3 codes of 1 and -1
                x = rng.choice(np.array([0x38, 0xB8], np.uint8), total)
                v = np.where(x == 0x38, 1, -1).astype(np.int32)
                xd = torch.from_numpy(x).cuda()
            else:
                v = workloads.uniform_i32(total, seed=nseg, lo=-4, hi=4)
                xd = torch.from_numpy(v).cuda().to(dtype)
            od = torch.from_numpy(off).cuda()
            want = oracle.segsum_i32(v, off)
            for form in (sr.F_ADAPTIVE_SEGMENTS, sr.F_BULK | 1, sr.F_BULK | 2, sr.F_BULK | 3, sr.F_BULK | 4, 0):
                for cfg in ({}, {"grid": 2}):
                    out = torch.full((nseg,), -99, dtype=sr.out_dtype(sr.dtype_code(xd), 0), device="cuda")
                    sr.reduce_sum_segmented(xd, od, out=out, config=sr.make_config(form, **cfg))
                    assert np.array_equal(out.cpu().numpy(), want), (nseg, total, form, cfg)
    assert sr.stream_status() == sr.OK


def _us(f, per=20):
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        f()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        for _ in range(per):
            f()
    best = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            g.replay()
        b.record()
        torch.cuda.synchronize()
        best.append(a.elapsed_time(b) / (5 * per) * 1e3)
    return sorted(best)[3]


def test_default_form_is_not_behind_the_ldg_kernel(sr):
    """Equal segments: measured 0.65 of the LDG kernel's time (1.3 with quarter chunks)."""
    nseg, length = 4096, 256
    x = torch.rand(nseg * length, device="cuda")
    off = torch.arange(nseg + 1, dtype=torch.int64, device="cuda") * length
    out = torch.empty(nseg, device="cuda")
    ldg = sr.make_config(sr.LAST_BLOCK, vec_bytes=32, unroll=8, block_threads=256)
    t = _us(lambda: sr.reduce_sum_segmented(x, off, out=out))
    t_ldg = _us(lambda: sr.reduce_sum_segmented(x, off, out=out, config=ldg))
    assert t < 1.05 * t_ldg, (t, t_ldg)
