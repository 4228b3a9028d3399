"""Runs of empty segments in the adaptive form and the TMA form: padded offsets,
keys that never occur.  All of a run lies at one element, so an unguarded split
by elements leaves it to one warp.  Lengths around the offsets window (32), the
second one, the blocks of 1024 segments and far beyond; runs before, among and
behind the data, at chunk starts and inside chunks; output filled beforehand,
so a segment that nothing writes shows; int32 exact, binary32 exact on small
integers."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

RUNS = [31, 32, 33, 62, 63, 64, 65, 95, 96, 97, 128, 1023, 1024, 1025, 2047, 2048, 2049, 5000, 40_000]


def _offsets(lens):
    off = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(np.asarray(lens, np.int64), out=off[1:])
    return off


def _check(sr, lens, first=0, seed=1, shift=0, finish=(0,), **cfg):
    off = _offsets(lens) + first
    n = max(int(off[-1]), 1)
    x = workloads.uniform_i32(n + shift, seed=seed, lo=-8, hi=8)
    od = torch.from_numpy(off).cuda()
    want = oracle.segsum_i32(np.ascontiguousarray(x[shift:]), off)
    for dtype in (torch.int32, torch.float32, torch.bfloat16):
        xd = torch.from_numpy(x).cuda().to(dtype)[shift:]
        for form in [sr.F_ADAPTIVE_SEGMENTS] + [sr.F_BULK | s for s in finish]:
            for flags in (0, sr.F_FP64_COMBINE | sr.F_KAHAN):
                code = sr.dtype_code(xd)
                out = torch.full((len(lens),), -7777, dtype=sr.out_dtype(code, flags), device="cuda")
                c = {k: v for k, v in cfg.items() if form != sr.F_ADAPTIVE_SEGMENTS or k == "grid"}
                sr.reduce_sum_segmented(xd, od, out=out, config=sr.make_config(form | flags, **c))
                got = out.cpu().numpy()
                bad = np.nonzero(got != want)[0]
                assert bad.size == 0, (dtype, form, flags, cfg, len(lens), bad[:5], got[bad[:5]], want[bad[:5]])


@pytest.mark.parametrize("run", RUNS)
def test_one_run(sr, run):
    rng = np.random.default_rng(run)
    short = list(rng.integers(0, 20, 500))
    z = [0] * run
    for lens in (z + short, short + z, short + z + short, z, z + [1], [1] + z, [5000] + z + [5000], [1024] + z + [1024] + z + [3]):
        _check(sr, lens, shift=int(rng.integers(0, 4)))


@pytest.mark.parametrize("shape", [{"grid": 1, "block_threads": 32}, {"grid": 3}, {"vec_bytes": 16, "unroll": 2, "stages": 3},
                                   {"vec_bytes": 32, "unroll": 8, "block_threads": 64}])
def test_many_runs(sr, shape):
    """Runs of random lengths at chunk starts, inside chunks of short and of long segments."""
    rng = np.random.default_rng(len(str(shape)))
    lens = []
    for k in range(40):
        lens += [0] * int(rng.choice(RUNS[:-1])) + list(rng.integers(0, rng.choice([3, 40, 2000]), int(rng.integers(1, 60))))
        if k % 8 == 0:  # the next run starts at a multiple of 2048 elements
            lens.append(-sum(lens) % 2048)
    _check(sr, lens, first=5, shift=3, finish=(1, 2, 3, 4), **shape)


def _ms(f):
    f()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    f()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b)


@pytest.mark.parametrize("where", ["behind", "before", "among", "all"])
def test_three_million_empty_segments_are_shared_by_the_grid(sr, where):
    """Results, and the time: at most ten times that of as many segments of one element
    (one warp alone takes a thousand times as long and more)."""
    m = 3 << 20
    data = np.full(1 << 16, 16, np.int64)
    z = np.zeros(m, np.int64)
    lens = {"behind": [data, z], "before": [z, data], "among": [data, z, data], "all": [z]}[where]
    lens = np.concatenate(lens)
    off = _offsets(lens)
    x = workloads.uniform_i32(max(int(off[-1]), 1), seed=2)
    xd, od = torch.from_numpy(x).cuda(), torch.from_numpy(off).cuda()
    ones = torch.arange(lens.size + 1, dtype=torch.int64, device="cuda")
    xo = torch.ones(lens.size, dtype=torch.int32, device="cuda")
    want = oracle.segsum_i32(x, off)
    for form in (sr.F_ADAPTIVE_SEGMENTS, sr.AUTO):
        out = torch.full((lens.size,), -7777, dtype=torch.int64, device="cuda")
        t = _ms(lambda: sr.reduce_sum_segmented(xd, od, variant=form, out=out))
        assert np.array_equal(out.cpu().numpy(), want), form
        t1 = _ms(lambda: sr.reduce_sum_segmented(xo, ones, variant=form, out=out))
        assert t < 10 * t1, (form, t, t1)
    assert sr.stream_status() == sr.OK
