// Argument block and kernel selection of the segmented sum, shared by the
// host planner (sr_segmented.cu) and the kernels (sr_segmented_kernels.cuh).
#pragma once
#include <cstdint>

#include "sr_kparams.h"

namespace sr {

constexpr int kErrBadOffsets = 4;  // the checked entry found offsets it may not read with

// TMA form: shared memory of one warp's strip table (one word per lane).  128
// bytes fit beside every ring that fits a CTA's shared memory without it (the
// tightest, 16 warps x 7 stages x 2 KiB, leaves 136 per warp).
constexpr int kStripTableBytes = 128;
// TMA form: a warp's piece is at least a chunk / kPieceParts, so the segments of
// a small input seldom cross a warp (100 segments of 30 elements: 8.3 us with
// pieces down to one vector, 6.9 now), and a whole chunk where segments average
// kLongMean bytes or more: a chunk then costs the same instructions however much of
// it is there, and more warps only add to them (4096 segments of 256 f32: 10.4 us
// with quarters, 9.0; equal ones 10.7, 5.3).  Shorter ones are summed by single
// lanes, for which whole chunks are too few warps (40,000 of 2: 5.2 us, 10.1; at a
// mean of 136 bytes 4096 to 7000 segments lose 3-9 % and 12,000 gain 2-14 %, at 168
// all but 4096 int32 ones gain).
constexpr int kPieceParts = 4;
constexpr int kLongMean = 160;

// Kernel argument block of the segmented sum (sr_segmented_kernels.cuh).
struct SegParams {
    const unsigned char* x;
    const int64_t* offsets;     // nseg + 1 entries, non-decreasing
    int64_t nseg;
    void* out;                  // nseg results
    unsigned char* carry_first; // W slots of 16 bytes (W = warps of the grid)
    unsigned char* carry_last;  // W slots of 16 bytes
    int64_t* last_seg;          // W entries: owned spanning segment or -1
    unsigned int* cnt;          // W self-resetting tickets (last-block form)
    int* err;
    float scale;
    int stage;
    int fp64;
    int stages;                 // TMA form: ring stages per warp
    uint64_t limit_ns;          // TMA form: bound of every mbarrier wait
    const int* bad;             // checked entry: nonzero = offsets invalid, read nothing (else NULL)
};

// Per-dtype segmented kernel selection, one function per kernel family and
// dtype (each in its own translation unit): the LDG form (which also returns
// the two-kernel form's second kernel), the dense variant, the TMA form.
const void* seg_ldg_f32(bool comp, int vec, int unroll, const void** fin);
const void* seg_dense_f32(bool comp, int vec, int unroll);
const void* seg_tma_f32(bool comp, int vec, int unroll);
const void* seg_ldg_i32(bool comp, int vec, int unroll, const void** fin);
const void* seg_dense_i32(bool comp, int vec, int unroll);
const void* seg_tma_i32(bool comp, int vec, int unroll);
const void* seg_ldg_bf16(bool comp, int vec, int unroll, const void** fin);
const void* seg_dense_bf16(bool comp, int vec, int unroll);
const void* seg_tma_bf16(bool comp, int vec, int unroll);
const void* seg_ldg_fp8(bool comp, int vec, int unroll, const void** fin);
const void* seg_dense_fp8(bool comp, int vec, int unroll);
const void* seg_tma_fp8(bool comp, int vec, int unroll);
// The warp-per-segment form, every dtype in one translation unit.
const void* seg_warp_f32(bool comp, int vec, int unroll);
const void* seg_warp_i32(bool comp, int vec, int unroll);
const void* seg_warp_bf16(bool comp, int vec, int unroll);
const void* seg_warp_fp8(bool comp, int vec, int unroll);
// The lane-per-segment form, in the same translation unit.
const void* seg_lane_f32(bool comp, int vec, int unroll);
const void* seg_lane_i32(bool comp, int vec, int unroll);
const void* seg_lane_bf16(bool comp, int vec, int unroll);
const void* seg_lane_fp8(bool comp, int vec, int unroll);

}  // namespace sr
