"""The form a segmented call takes when the caller names none, either side of
the segment counts where it changes, against the oracle: every dtype, plain and
compensated, and the resolved plan, which is itself a valid configuration."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

EPS32 = 2.0 ** -23


@pytest.mark.parametrize("nseg", [4095, 4096, 4097, 32767, 32768])
def test_default_form(sr, nseg):
    rng = np.random.default_rng(nseg)
    lens = rng.integers(0, 200, nseg)
    lens[rng.random(nseg) < 0.01] = 20_000  # a few long ones
    off = np.zeros(nseg + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    n = int(off[-1])
    od = torch.from_numpy(off).cuda()
    x = workloads.uniform_f32(n, seed=1)
    sabs, ex = oracle.segsum_abs_f32(x, off), oracle.segexact_f32(x, off)
    xi = workloads.uniform_i32(n, seed=1)
    bits = workloads.to_bf16_bits(x)
    dec = np.frombuffer((bits.astype(np.uint32) << 16).tobytes(), np.float32)
    for back in (False, True):  # the default, then the plan it resolves to
        def cfg(dt, flags=0):
            c = sr.make_config(sr.AUTO | flags)
            return sr.plan_segmented(nseg, dt, c) if back else c
        got = sr.reduce_sum_segmented(torch.from_numpy(xi).cuda(), od, config=cfg(sr.I32)).cpu().numpy()
        assert np.array_equal(got, oracle.segsum_i32(xi, off))
        xd = torch.from_numpy(x).cuda()
        for flags in (0, sr.F_KAHAN):
            got = sr.reduce_sum_segmented(xd, od, config=cfg(sr.F32, flags)).cpu().numpy()
            assert np.all(np.abs(got - ex) <= 4 * EPS32 * sabs + 1e-30), (back, flags)
        got = sr.reduce_sum_segmented(torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16), od,
                                      config=cfg(sr.BF16)).cpu().numpy()
        assert np.all(np.abs(got - oracle.segexact_f32(dec, off)) <=
                      4 * EPS32 * oracle.segsum_abs_f32(dec, off) + 1e-30)
    adaptive = bool(sr.plan_segmented(nseg, sr.F32).variant & sr.F_ADAPTIVE_SEGMENTS)
    assert adaptive == (4096 <= nseg < 32768)
    # a stage, a grid or a shape keeps the flat split's LDG form below 32768 segments
    for c in (sr.make_config(sr.TWO_KERNEL), sr.make_config(grid=64), sr.make_config(unroll=4)):
        assert not sr.plan_segmented(nseg, sr.F32, c).variant & sr.F_ADAPTIVE_SEGMENTS
    assert sr.stream_status() == sr.OK
