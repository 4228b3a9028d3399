"""The TMA form's strip kernel at the sizes where it can go wrong: segments
around a vector, a strip (1/32 of a chunk) and a chunk; windows of 32 offsets
filled with empty segments; chunks that begin with short segments and end in a
long one and the other way round; every dtype, aligned and misaligned, one CTA
and the default grid.  int32 is exact; a binary32 result of additions in any
order is within the plain gate 4 eps32 sum|x| used by the other segmented tests.
"""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

BULK = 0x400
EPS32 = 2.0 ** -23
U = 2.0 ** -24


def _offsets(lens):
    off = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(np.asarray(lens, np.int64), out=off[1:])
    return off


def _layout(name, elem):
    """Segment lengths over a few chunks of 4096 bytes, for elements of `elem` bytes."""
    ce = 4096 // elem
    se, ev = ce // 32, 16 // elem
    rng = np.random.default_rng(elem)
    if name == "vector":
        return [k for k in (1, 2, ev - 1, ev, ev + 1) for _ in range(max(1, 3 * ce // max(k, 1) // 5))]
    if name == "strip":
        return [k for k in (se - 1, se, se + 1, 2 * se - 1, 2 * se + 1) for _ in range(40)]
    if name == "chunk":
        return [k for k in (ce - 1, ce, ce + 1, 2 * ce, 5) for _ in range(4)]
    if name == "empty_windows":  # runs of 20 to 100 empty segments between short and long ones
        return [v for k in range(60) for v in [0] * int(rng.integers(20, 100)) + [int(rng.integers(1, 2 * se))]]
    if name == "short_then_long":  # more than one window of short ones, then a long one
        return [v for _ in range(6) for v in [int(rng.integers(1, ev + 2)) for _ in range(45)] + [int(ce + rng.integers(0, ce))]]
    assert name == "long_then_short"
    return [v for _ in range(12) for v in [int(rng.integers(se, ce))] + [int(rng.integers(0, ev + 2)) for _ in range(70)]]


@pytest.mark.parametrize("name", ["vector", "strip", "chunk", "empty_windows", "short_then_long", "long_then_short"])
def test_strip_edges(sr, name):
    for elem in (4, 2, 1):
        off = _offsets(_layout(name, elem))
        n = int(off[-1])
        od = torch.from_numpy(off).cuda()
        for shift in (0, 1, 3):
            for shape in ({}, {"grid": 1, "block_threads": 32}, {"vec_bytes": 16, "unroll": 2, "stages": 3},
                          {"vec_bytes": 32, "unroll": 8, "stages": 2, "block_threads": 64}):
                stage = (1, 2, 3, 4)[(shift + len(shape)) % 4]
                if elem == 4:
                    xi = workloads.uniform_i32(n + shift, seed=shift)
                    xd = torch.from_numpy(xi).cuda()[shift:]
                    got = sr.reduce_sum_segmented(xd, od, config=sr.make_config(stage | BULK, **shape)).cpu().numpy()
                    assert np.array_equal(got, oracle.segsum_i32(xi[shift:], off)), (shift, shape)
                x = workloads.uniform_f32(n + shift, seed=shift + 5)
                if elem == 4:
                    xd, dec, scale = torch.from_numpy(x).cuda()[shift:], x[shift:], 0.0
                elif elem == 2:
                    bits = workloads.to_bf16_bits(x)
                    xd = torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)[shift:]
                    dec, scale = np.frombuffer((bits.astype(np.uint32) << 16).tobytes(), np.float32)[shift:], 0.0
                else:
                    codes, scale = workloads.to_e4m3_codes(x)
                    xd = torch.from_numpy(codes).cuda()[shift:]
                    dec = (torch.from_numpy(codes).view(torch.float8_e4m3fn).float() * scale).numpy()[shift:]
                ex = oracle.segexact_f32(np.ascontiguousarray(dec), off)
                sabs = oracle.segsum_abs_f32(np.ascontiguousarray(dec), off)
                for flags in (0, sr.F_KAHAN):
                    got = sr.reduce_sum_segmented(xd, od, config=sr.make_config(stage | BULK | flags, scale=scale,
                                                                                **shape)).cpu().numpy()
                    # FP8: each decoded value times the scale is rounded once in `dec`, and the result's own
                    # product with the scale once more
                    tol = (4 * EPS32 if not flags else 2 * U) * sabs + (4 * U * sabs if elem == 1 else 0.0)
                    tol = tol + np.diff(off) * U * U * sabs + 1e-30
                    bad = np.nonzero(np.abs(got.astype(np.float64) - ex) > tol)[0]
                    assert bad.size == 0, (elem, shift, shape, flags, bad[:5], got[bad[:5]], ex[bad[:5]])
    assert sr.stream_status() == sr.OK


def test_infinities_and_nans_stay_in_their_segment(sr):
    """Elements beside a boundary are cut off by masks, never multiplied away."""
    lens = [7, 0, 33, 5, 1100, 3, 64, 2, 2, 900, 31, 32, 33]
    off = _offsets(lens * 3)
    x = workloads.uniform_f32(int(off[-1]), seed=1)
    hit = {2: np.inf, 4: np.nan, 8: -np.inf, 20: np.inf, 30: np.nan}
    for s, v in hit.items():
        x[off[s]] = v
        x[off[s + 1] - 1] = v
    got = sr.reduce_sum_segmented(torch.from_numpy(x).cuda(), torch.from_numpy(off).cuda(),
                                  config=sr.make_config(sr.LAST_BLOCK | BULK)).cpu().numpy()
    for s in range(off.size - 1):
        if s in hit:
            assert np.isnan(got[s]) if np.isnan(hit[s]) else got[s] == hit[s], s
        else:
            seg = x[off[s]:off[s + 1]].astype(np.float64)
            assert abs(got[s] - seg.sum()) <= 4 * EPS32 * np.abs(seg).sum(), s


def test_ring_that_fills_the_sm(sr):
    """A ring that two CTAs per SM just hold: the strip tables take a stage's
    place, and a grid.sync() grid of two CTAs per SM still runs."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    off = workloads.segment_offsets(3000, 1 << 22, seed=3, median=512, sigma=1.5, lo=0, hi=1 << 16)
    x = workloads.uniform_i32(int(off[-1]), seed=3)
    for shape in ({"vec_bytes": 16, "unroll": 4, "stages": 7, "block_threads": 256},
                  {"vec_bytes": 32, "unroll": 4, "stages": 4, "block_threads": 224}):
        got = sr.reduce_sum_segmented(torch.from_numpy(x).cuda(), torch.from_numpy(off).cuda(),
                                      config=sr.make_config(sr.GRID_SYNC | BULK, grid=2 * sms, **shape)).cpu().numpy()
        assert np.array_equal(got, oracle.segsum_i32(x, off)), shape
