"""Segmented sums of constant data, whose rounding errors all have one sign: any
plain chain of binary32 additions that grows with the input leaves the plain
gate 4 eps32 sum|x| here.  Segments of many chunks of the strip kernel, of one
warp and of every warp of the grid; each result against length x value, exact
in binary64."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

EPS32 = 2.0 ** -23


@pytest.mark.parametrize("nseg,length", [(4200, 60_000), (100, 1 << 21), (1, (1 << 28) + 3)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_constant_data_stays_within_the_gate(sr, nseg, length, dtype):
    off = torch.arange(nseg + 1, dtype=torch.int64, device="cuda") * length
    x = torch.full((nseg * length,), 0.1, dtype=dtype, device="cuda")
    want = float(x[0]) * length
    variants = [sr.F_ADAPTIVE_SEGMENTS, sr.F_BULK | sr.LAST_BLOCK, sr.F_BULK | sr.TWO_KERNEL, sr.F_BULK | sr.GRID_SYNC]
    if nseg >= 4096:
        variants.append(sr.AUTO)
    for v in variants:
        got = sr.reduce_sum_segmented(x, off, variant=v).double().cpu().numpy()
        assert np.max(np.abs(got - want)) <= 4 * EPS32 * want, (v, np.max(np.abs(got - want)) / (EPS32 * want))
    assert sr.stream_status() == sr.OK


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite_values_in_a_long_segment(sr, value):
    """One such value in a segment of many chunks is its sum; two opposite infinities are NaN."""
    n = 1 << 22
    off = torch.tensor([0, 5, n - 7, n], dtype=torch.int64, device="cuda")
    x = torch.ones(n, dtype=torch.float32, device="cuda")
    x[n // 3] = value
    for v in (sr.F_ADAPTIVE_SEGMENTS, sr.F_BULK | sr.TWO_KERNEL):
        for grid in (0, 1):
            got = sr.reduce_sum_segmented(x, off, config=sr.make_config(v, grid=grid)).cpu().numpy()
            assert got[0] == 5 and got[2] == 7
            assert np.isnan(got[1]) if np.isnan(value) else got[1] == value
            y = x.clone()
            y[2 * n // 3] = -value
            assert np.isnan(sr.reduce_sum_segmented(y, off, config=sr.make_config(v, grid=grid)).cpu().numpy()[1])
