"""int32 segments with nothing asked for: the finish is atomic (exact in any
order) below 2^19 segments in both forms the default takes, by tickets from
there on; results exact, whatever the output held before."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nseg", [4095, 4096, 10_000, 32_767, 32_768, (1 << 19) - 1, 1 << 19])
def test_int32_default_finish(sr, nseg):
    stage = sr.plan_segmented(nseg, sr.I32).variant & 0xF
    assert stage == (sr.ATOMIC if nseg < 1 << 19 else sr.LAST_BLOCK)
    off = workloads.random_segment_offsets(nseg, 60, seed=nseg)
    x = workloads.uniform_i32(int(off[-1]), seed=3)
    out = torch.full((nseg,), -7, dtype=torch.int64, device="cuda")
    for _ in range(2):
        sr.reduce_sum_segmented(torch.from_numpy(x).cuda(), torch.from_numpy(off).cuda(), out=out)
        assert np.array_equal(out.cpu().numpy(), oracle.segsum_i32(x, off))
