// Segmented (batched) sum: out[s] = sum of x[offsets[s] .. offsets[s+1]).
// Kernel templates, instantiated per input dtype by sr_segmented_<dtype>.cu.
//
// Work split of the flat forms: the concatenated range [offsets[0], offsets[nseg]) is cut into
// W equal, vector-aligned pieces of E elements, one per warp of the grid, so
// the load is balanced whatever the segment lengths.  Segment s is *owned*
// by the warp whose piece contains offsets[s].  Each warp
//   - sums the continuation of the segment that started before its piece
//     (its "first carry"),
//   - sums every segment it owns; a segment that ends inside the piece is
//     written to out directly, the one that runs past the end of the piece
//     leaves a "last carry".
// A segment spanning warps w_o..w_e is then finished as
//   out[s] = carry_last[w_o] + sum_{w = w_o+1..w_e} carry_first[w]
// in that fixed order (deterministic), after a grid-level join of one of four
// forms (the paper's Section VII-E barrier choice applied to the batch):
//   two-kernel  : a second kernel does every finish (implicit barrier);
//   grid.sync   : cooperative kernel, finishes after grid.sync();
//   last-block  : per-segment ticket; the last contributing warp finishes;
//   atomic      : spanning pieces atomically added into out (zeroed first).
// The end of this file holds two forms without that split: whole segments
// per warp and whole segments per thread (no carries, no grid stage).
#pragma once

#include <type_traits>

#include "sr_device.cuh"
#include "sr_kparams.h"
#include "sr_segparams.h"

namespace sr {

template <int DT> struct SegElem { static constexpr int v = 4; };
template <> struct SegElem<kDtBF16> { static constexpr int v = 2; };
template <> struct SegElem<kDtFP8> { static constexpr int v = 1; };

// ------------------------------------------------------------ helpers
// First s in [0, nseg] with offsets[s] >= key (nseg if none).  Warp-wide:
// each round, 32 samples shrink the interval 32-fold.
__device__ __forceinline__ void lb_round(const int64_t* off, int64_t key, int lane, int64_t& lo, int64_t& hi) {
    if (hi - lo <= 32) return;
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t i = lo + (int64_t)lane * step;
    const bool pred = (i < hi) ? (__ldg(off + i) >= key) : true;
    const unsigned m = __ballot_sync(0xffffffffu, pred);
    if (m == 0) {
        lo = lo + 31 * step + 1;
    } else {
        const int k = __ffs(m) - 1;
        const int64_t ik = lo + (int64_t)k * step;
        hi = ik < hi ? ik : hi;
        if (k > 0) lo = lo + (int64_t)(k - 1) * step + 1;
    }
}
// hi - lo <= 32 here.  With exactly 32 candidates left, every lane may hold
// an offset below the key: the ballot is then empty and the answer is hi.
__device__ __forceinline__ int64_t lb_final(const int64_t* off, int64_t key, int lane, int64_t lo, int64_t hi) {
    const int64_t i = lo + lane;
    const bool pred = (i < hi) ? (__ldg(off + i) >= key) : true;
    const unsigned m = __ballot_sync(0xffffffffu, pred);
    if (m == 0) return hi;
    const int64_t r = lo + (__ffs(m) - 1);
    return r < hi ? r : hi;
}
__device__ __forceinline__ int64_t warp_lower_bound(const int64_t* off, int64_t nseg, int64_t key, int lane) {
    int64_t lo = 0, hi = nseg;  // answer in [lo, hi]
    while (hi - lo > 32) lb_round(off, key, lane, lo, hi);
    return lb_final(off, key, lane, lo, hi);
}

// The first s in [0, nseg] with offsets[s] >= key, and the offsets around it.
// On return lane k holds offsets[wb + k] in `win` (INT64_MAX past offsets[nseg])
// and the answer r lies in [wb, wb + 30], so offsets[r] and offsets[r + 1] are
// in the window.  The first probe spreads the lanes at power-of-two distances
// around `guess`, the answer for equal segments: for layouts near it that is
// one round of loads instead of log32(nseg) (whole warp calls).  `meanwhile` runs
// when the last round is on its way: bulk traffic belongs there, since earlier
// rounds would queue behind it.
template <class F>
__device__ __forceinline__ int64_t warp_search(const int64_t* off, int64_t nseg, int64_t key, int64_t guess, int lane,
                                               int64_t& wb, int64_t& win, F&& meanwhile) {
    int64_t lo = 0, hi = nseg;  // the answer is in [lo, hi]
    if (nseg > 30) {
        const int64_t i = lane < 16 ? guess - (1 << (15 - lane)) : guess + (1 << (lane - 16)) - 1;
        const bool pred = i >= nseg || (i >= 0 && __ldg(off + i) >= key);
        const unsigned m = __ballot_sync(0xffffffffu, pred);
        const int k = m ? __ffs(m) - 1 : 32;
        const int64_t below = __shfl_sync(0xffffffffu, i, k > 0 ? k - 1 : 0);
        const int64_t at = __shfl_sync(0xffffffffu, i, k < 32 ? k : 31);
        if (k > 0 && below >= 0) lo = below + 1;
        if (k < 32 && at < nseg) hi = at;
    }
    while (hi - lo > 30) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t i = lo + (int64_t)lane * step;
        const bool pred = (i < hi) ? (__ldg(off + i) >= key) : true;
        const unsigned m = __ballot_sync(0xffffffffu, pred);
        if (m == 0) {
            lo = lo + 31 * step + 1;
        } else {
            const int k = __ffs(m) - 1;
            const int64_t ik = lo + (int64_t)k * step;
            hi = ik < hi ? ik : hi;
            if (k > 0) lo = lo + (int64_t)(k - 1) * step + 1;
        }
    }
    wb = lo;
    win = (lo + lane <= nseg) ? __ldg(off + lo + lane) : INT64_MAX;
    meanwhile();
    return lo + __ffs(__ballot_sync(0xffffffffu, lo + lane >= hi || win >= key)) - 1;
}

// Bits j of a PV-bit mask with a <= j < b (a and b clamped to [0, PV]).
template <int PV> __device__ __forceinline__ uint32_t run_mask(int64_t a, int64_t b) {
    const int ja = a <= 0 ? 0 : (a >= PV ? PV : (int)a);
    const int jb = b <= 0 ? 0 : (b >= PV ? PV : (int)b);
    const uint32_t below_b = jb >= 32 ? 0xffffffffu : (1u << jb) - 1u;
    const uint32_t below_a = ja >= 32 ? 0xffffffffu : (1u << ja) - 1u;
    return below_b & ~below_a;
}

// Sum of a lane's W word accumulators as a pairwise tree (log2 W dependent adds).
template <class A, int W> __device__ __forceinline__ A sum_words(const A (&acc)[W]) {
    A t[W];
#pragma unroll
    for (int k = 0; k < W; ++k) t[k] = acc[k];
#pragma unroll
    for (int h = 1; h < W; h <<= 1) {
#pragma unroll
        for (int k = 0; k + h < W; k += 2 * h) t[k] = Op<A>::add(t[k], t[k + h]);
    }
    return t[0];
}

// Element j of a vector held as 32-bit words (the masked slow path; j is a
// compile-time constant after unrolling).
template <int DT, class A> __device__ __forceinline__ void acc_vec_elem(A& a, const uint32_t* r, int j);
template <> __device__ __forceinline__ void acc_vec_elem<kDtI32, long long>(long long& a, const uint32_t* r, int j) {
    a += (long long)(int)r[j];
}
template <class A> __device__ __forceinline__ void acc_vec_elem_f32(A& a, const uint32_t* r, int j) {
    acc_add_f(a, __uint_as_float(r[j]));
}
template <class A> __device__ __forceinline__ void acc_vec_elem_bf16(A& a, const uint32_t* r, int j) {
    const uint32_t w = r[j >> 1];
    acc_add_f(a, __uint_as_float((j & 1) ? (w & 0xffff0000u) : (w << 16)));
}
template <class A> __device__ __forceinline__ void acc_vec_elem_fp8(A& a, const uint32_t* r, int j) {
    const uint32_t w = r[j >> 2];
    __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)((w >> (8 * (j & 3))) & 0xffu), __NV_E4M3);
    acc_add_f(a, __half2float(*reinterpret_cast<__half*>(&h)));
}
template <> __device__ __forceinline__ void acc_vec_elem<kDtF32, float>(float& a, const uint32_t* r, int j) { acc_vec_elem_f32(a, r, j); }
template <> __device__ __forceinline__ void acc_vec_elem<kDtF32, Pair>(Pair& a, const uint32_t* r, int j) { acc_vec_elem_f32(a, r, j); }
template <> __device__ __forceinline__ void acc_vec_elem<kDtBF16, float>(float& a, const uint32_t* r, int j) { acc_vec_elem_bf16(a, r, j); }
template <> __device__ __forceinline__ void acc_vec_elem<kDtBF16, Pair>(Pair& a, const uint32_t* r, int j) { acc_vec_elem_bf16(a, r, j); }
template <> __device__ __forceinline__ void acc_vec_elem<kDtFP8, float>(float& a, const uint32_t* r, int j) { acc_vec_elem_fp8(a, r, j); }
template <> __device__ __forceinline__ void acc_vec_elem<kDtFP8, Pair>(Pair& a, const uint32_t* r, int j) { acc_vec_elem_fp8(a, r, j); }

// ---------------------------------------------------- output and carries
__device__ __forceinline__ void seg_out(const SegParams& p, int64_t s, long long v) {
    reinterpret_cast<long long*>(p.out)[s] = v;
}
template <class A> __device__ __forceinline__ void seg_out(const SegParams& p, int64_t s, A v) {
    if (p.fp64) reinterpret_cast<double*>(p.out)[s] = __dmul_rn(to_double(v), (double)p.scale);
    else reinterpret_cast<float*>(p.out)[s] = __fmul_rn(to_float(v), p.scale);
}
__device__ __forceinline__ void seg_out_d(const SegParams& p, int64_t s, double v) {
    reinterpret_cast<double*>(p.out)[s] = __dmul_rn(v, (double)p.scale);
}
__device__ __forceinline__ void seg_atomic(const SegParams& p, int64_t s, long long v) {
    atomicAdd(reinterpret_cast<unsigned long long*>(p.out) + s, (unsigned long long)v);
}
template <class A> __device__ __forceinline__ void seg_atomic(const SegParams& p, int64_t s, A v) {
    if (p.fp64) atomicAdd(reinterpret_cast<double*>(p.out) + s, __dmul_rn(to_double(v), (double)p.scale));
    else atomicAdd(reinterpret_cast<float*>(p.out) + s, __fmul_rn(to_float(v), p.scale));
}

template <class A> __device__ __forceinline__ void carry_store(const SegParams& p, unsigned char* arr, int64_t w, A v) {
    unsigned char* slot = arr + w * 16;
    if (p.fp64) *reinterpret_cast<double*>(slot) = to_double(v);
    else *reinterpret_cast<A*>(slot) = v;
}
template <> __device__ __forceinline__ void carry_store<long long>(const SegParams& p, unsigned char* arr, int64_t w,
                                                                   long long v) {
    (void)p;
    *reinterpret_cast<long long*>(arr + w * 16) = v;
}

template <class P> __device__ __forceinline__ P carry_load(const unsigned char* arr, int64_t w) {
    const unsigned char* s = arr + w * 16;
    if constexpr (std::is_same<P, Pair>::value) {
        float2 v = __ldcg(reinterpret_cast<const float2*>(s));
        return Pair{v.x, v.y};
    } else {
        return __ldcg(reinterpret_cast<const P*>(s));
    }
}

// A running sum of partial sums whose number grows with the input.  A plain
// binary32 chain of k same-sign additions errs by up to k u |S| (64 additions of
// 0.1f exceed 4 eps32 |S|), so there it carries the rounding errors along
// (TwoSum); int64 is exact, pairs carry theirs already, and binary64 has room.
template <class A> struct RunSum {
    A v;
    __device__ __forceinline__ static RunSum of(A x) { return RunSum{x}; }
    __device__ __forceinline__ void add(A x) { v = Op<A>::add(v, x); }
    __device__ __forceinline__ A total() const { return v; }
    __device__ __forceinline__ A only() const { return v; }  // the sum when nothing was added to it
};
template <> struct RunSum<float> {
    float s, c;
    __device__ __forceinline__ static RunSum of(float x) { return RunSum{x, 0.f}; }
    __device__ __forceinline__ void add(float x) {
        float t, e;
        two_sum(s, x, t, e);
        s = t;
        c = __fadd_rn(c, e);
    }
    // an infinite sum leaves a NaN correction
    __device__ __forceinline__ float total() const { return c == c ? __fadd_rn(s, c) : s; }
    __device__ __forceinline__ float only() const { return s; }
};

// Finish a spanning segment s owned by warp w_o, ending in warp w_e (whole
// warp calls; fixed order, so the result does not depend on which warp runs it).
// WIDE: eight loads in flight, for a long segment has thousands of carries (one of
// 2^24 elements 22.2 -> 20.0 us), added as a tree and those trees' sums as a RunSum.
// The LDG kernel keeps the plain loop: with the wide one its hot loop got fewer
// registers (10,000 lognormal segments at 32 B x 4: 168 -> 205 us).
template <class P, bool WIDE> __device__ __forceinline__ void finish_span_typed(const SegParams& p, int64_t s,
                                                                                int64_t w_o, int64_t w_e, int lane) {
    P acc = Op<P>::zero(), own = Op<P>::zero();
    int64_t w = w_o + 1 + lane;
    if constexpr (WIDE) {
        own = carry_load<P>(p.carry_last, w_o);  // one trip together with the others
        RunSum<P> sum = RunSum<P>::of(acc);
        for (; w + 7 * 32 <= w_e; w += 8 * 32) {
            P c[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) c[k] = carry_load<P>(p.carry_first, w + 32 * k);
            sum.add(sum_words<P, 8>(c));
        }
        for (; w <= w_e; w += 32) sum.add(carry_load<P>(p.carry_first, w));
        acc = sum.total();
    } else {
        for (; w <= w_e; w += 32) acc = Op<P>::add(acc, carry_load<P>(p.carry_first, w));
    }
    acc = warp_reduce(acc);
    if (lane == 0) {
        P total = Op<P>::add(WIDE ? own : carry_load<P>(p.carry_last, w_o), acc);
        if constexpr (std::is_same<P, double>::value) seg_out_d(p, s, total);
        else seg_out(p, s, total);
    }
}
template <class A, bool WIDE> __device__ __forceinline__ void finish_span(const SegParams& p, int64_t s, int64_t w_o,
                                                                          int64_t w_e, int lane) {
    if constexpr (std::is_same<A, long long>::value) {
        finish_span_typed<long long, WIDE>(p, s, w_o, w_e, lane);
    } else {
        if (p.fp64) finish_span_typed<double, WIDE>(p, s, w_o, w_e, lane);
        else finish_span_typed<A, WIDE>(p, s, w_o, w_e, lane);
    }
}

// Per-segment ticket of the last-block form: every contributing warp
// arrives once; the last one finishes the segment and resets the ticket.
template <class A, bool WIDE> __device__ __forceinline__ void span_arrive(const SegParams& p, int64_t s, int64_t w_o,
                                                                          int64_t w_e, int lane) {
    unsigned t = 0;
    if (lane == 0) {
        __threadfence();
        t = atomicAdd(p.cnt + w_o, 1u);
    }
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t == (unsigned)(w_e - w_o)) {
        __threadfence();
        finish_span<A, WIDE>(p, s, w_o, w_e, lane);
        if (lane == 0) atomicExch(p.cnt + w_o, 0u);
    }
}

// ------------------------------------------------------------- main kernel
// One warp walks its piece [lo, hi) in element order: a scalar head up to the
// vector alignment, rows of 32 lane vectors (loads issued UNROLL rows ahead,
// independently of where segments end), and a scalar tail.  The current
// segment and its end travel with the walk; a row that contains no boundary
// is accumulated whole, a row that does takes a masked per-element path and
// emits each segment that ends in it — the load pipeline never drains at a
// boundary.
constexpr int kScanMin = 3;  // boundaries in a row from which the warp-wide pass pays

template <int DT, bool COMP, int VB, int UNROLL, bool DENSE>
__global__ void __launch_bounds__(512, 1) seg_kernel(const SegParams p) {
    using A = typename Acc<DT, COMP>::T;
    constexpr int EB = SegElem<DT>::v;
    constexpr int PV = VB / EB;  // elements per lane vector
    constexpr int W = VB / 4;    // 32-bit words per lane vector
    constexpr int RW = 32 * PV;  // elements per row
    grid_dependency_wait();
    allow_dependents();
    if (p.bad != nullptr && __ldcg(p.bad) != 0) return;  // offsets failed the check: read nothing
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t Wn = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t base = __ldg(p.offsets);
    const int64_t N = __ldg(p.offsets + p.nseg) - base;
    int64_t E = (N + Wn - 1) / Wn;
    E = ((E + PV - 1) / PV) * PV;
    if (E < PV) E = PV;
    const int64_t lo = base + (w * E < N ? w * E : N);
    const int64_t hi = base + ((w + 1) * E < N ? (w + 1) * E : N);
    const int64_t next_lo = (w == Wn - 1) ? INT64_MAX : base + (w + 1) * E;

    // geometry of the piece: scalar head [lo, a0), vector rows [a0, hi_al), scalar tail [hi_al, hi)
    const uintptr_t addr = reinterpret_cast<uintptr_t>(p.x) + (uintptr_t)lo * EB;
    int64_t a0 = lo + (int64_t)(((uintptr_t)VB - addr % VB) % VB) / EB;
    if (a0 > hi) a0 = hi;
    const int64_t nvec = (hi - a0) / PV;
    const int64_t hi_al = a0 + nvec * PV;
    const int64_t nrows = (nvec + 31) / 32;
    const unsigned char* body = p.x + a0 * EB;

    // first batch of rows in flight before the segment search
    uint32_t buf[UNROLL][W];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
        const int64_t v = (int64_t)u * 32 + lane;
        if (v < nvec) ldg_vec(body + v * VB, buf[u]);
    }

    const int64_t s_begin = warp_lower_bound(p.offsets, p.nseg, base + w * E, lane);
    // stream state (warp-uniform): segment `cur` = [cur_start, cur_end)
    int64_t cur = s_begin;
    if (lo < hi && s_begin > 0 && __ldg(p.offsets + s_begin) > lo) cur = s_begin - 1;  // continuation
    int64_t wb = cur + 1;  // offsets window: lane k holds offsets[wb + k]
    int64_t win = (wb + lane <= p.nseg) ? __ldg(p.offsets + wb + lane) : INT64_MAX;
    int64_t cur_start = (cur < p.nseg) ? __ldg(p.offsets + cur) : INT64_MAX;
    int64_t cur_end = (cur < p.nseg) ? __shfl_sync(0xffffffffu, win, 0) : INT64_MAX;
    int64_t spanning = -1;
    A acc[W];  // one accumulator per 32-bit word of the lane vector
#pragma unroll
    for (int k = 0; k < W; ++k) acc[k] = Op<A>::zero();

    // emit the current segment's piece and move to the next segment
    auto emit_advance = [&]() {
        A v = warp_reduce(sum_words<A, W>(acc));
#pragma unroll
        for (int k = 0; k < W; ++k) acc[k] = Op<A>::zero();
        const int64_t s = cur;
        if (cur_start < lo) {  // continuation of a segment owned by an earlier warp
            if (p.stage == kStageAtomic) {
                if (lane == 0) seg_atomic(p, s, v);
            } else {
                if (lane == 0) carry_store(p, p.carry_first, w, v);
                if (p.stage == kStageLastBlock)
                    span_arrive<A, false>(p, s, (cur_start - base) / E, (cur_end - 1 - base) / E, lane);
            }
        } else if (cur_end <= hi) {  // owned and complete
            if (lane == 0) seg_out(p, s, v);
        } else {  // owned, runs past this piece
            spanning = s;
            if (p.stage == kStageAtomic) {
                if (lane == 0) seg_atomic(p, s, v);
            } else {
                if (lane == 0) carry_store(p, p.carry_last, w, v);
                if (p.stage == kStageLastBlock) span_arrive<A, false>(p, s, w, (cur_end - 1 - base) / E, lane);
            }
        }
        cur += 1;
        cur_start = cur_end;
        if (cur >= p.nseg) {
            cur_end = INT64_MAX;
            return;
        }
        if (cur + 1 - wb >= 32) {
            wb = cur + 1;
            win = (wb + lane <= p.nseg) ? __ldg(p.offsets + wb + lane) : INT64_MAX;
        }
        cur_end = __shfl_sync(0xffffffffu, win, (int)(cur + 1 - wb));
    };

    // A row [c0, c1) in which segments end, every boundary resolved in one
    // warp-wide pass: each lane splits its vector at the boundary it holds
    // (head before, tail from it on), a segmented inclusive scan over the lanes
    // (flag = the lane holds a boundary) yields the run open at the end of
    // every lane, and the lane holding boundary j emits the segment that ends
    // there: cur itself for j = 0 (with the rows before folded in; cur must be
    // owned by this warp, a continuation takes the per-segment path), an owned
    // segment complete inside the row for j >= 1.  The run open at the row's
    // end becomes the next segment's carry.  Applies when the row holds at
    // least kScanMin boundaries (below that one warp reduction per boundary is
    // cheaper than the pass's fixed ~17 shuffle rounds), no lane holds two,
    // and the offsets window already holds all of them; returns false, having
    // changed nothing, otherwise (no load is spent on a row that may fail).
    auto row_scan = [&](int64_t c0, int64_t c1, int64_t e0, bool valid, const uint32_t (&r_words)[W]) -> bool {
        if (cur_start < lo) return false;  // cur continues an earlier warp's segment: per-segment path
        const int kb = (int)(cur + 1 - wb);  // window lane of the row's first boundary
        const bool is_b = lane >= kb && win < c1;  // the row's boundaries: lanes kb .. kb + m - 1
        const unsigned bm = __ballot_sync(0xffffffffu, is_b);
        if (bm & 0x80000000u) return false;  // more boundaries may follow beyond the window
        const int m = __popc(bm);
        if (m < kScanMin) return false;
        const int tl = is_b ? (int)((win - c0) / PV) : -1;  // lane of the row holding boundary
        const int tl_next = __shfl_down_sync(0xffffffffu, tl, 1);
        if (__any_sync(0xffffffffu, is_b && lane < 31 && tl_next == tl)) return false;  // two in one lane
        const unsigned tmask = __reduce_or_sync(0xffffffffu, is_b ? (1u << tl) : 0u);
        const bool has_b = (tmask >> lane) & 1u;
        const int bj = __popc(tmask & ((1u << lane) - 1u));  // this lane's boundary among the row's
        const int64_t bpos = __shfl_sync(0xffffffffu, win, (kb + bj) & 31);
        const int q = has_b ? (int)(bpos - e0) : PV;  // elements j < q precede the boundary
        A head = Op<A>::zero(), tail = Op<A>::zero();
        if (valid) {
            const int jv = (c1 - e0 < PV) ? (int)(c1 - e0) : PV;  // elements of the lane inside the row
#pragma unroll
            for (int j = 0; j < PV; ++j) {
                if (j < jv) {
                    if (j < q) acc_vec_elem<DT>(head, r_words, j);
                    else acc_vec_elem<DT>(tail, r_words, j);
                }
            }
        }
        // segmented inclusive scan of the open runs over the lanes; before the
        // step with distance d a lane's partial covers lanes [lane - d + 1,
        // lane], which holds a boundary exactly when tmask has a bit there
        A x = has_b ? tail : head;
        const unsigned upto = (2u << lane) - 1u;  // lanes 0 .. lane (wraps to all ones at 31)
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const A xo = Op<A>::shfl_up(x, d);
            const int first = lane - d + 1 > 0 ? lane - d + 1 : 0;
            const bool f = (tmask & upto & ~((1u << first) - 1u)) != 0u;
            if (lane >= d && !f) x = Op<A>::add(xo, x);
        }
        A prev = Op<A>::shfl_up(x, 1);  // the run open at the end of the previous lane
        if (lane == 0) prev = Op<A>::zero();
        const A closed = Op<A>::add(prev, head);  // the segment ending at this lane's boundary
        const A open_end = Op<A>::shfl(x, 31);   // the run open at the row's end
        const int64_t last_pos = __shfl_sync(0xffffffffu, win, (kb + m - 1) & 31);
        const int64_t cur0 = cur;
        // owned segments complete inside the row (boundaries j >= 1)
        if (has_b && bj >= 1) seg_out(p, cur0 + bj, closed);
        // segment cur, owned by this warp and complete: the rows before this
        // one (acc, per lane) plus its part of this row
        const A first = Op<A>::shfl(closed, __ffs(tmask) - 1);
        A t = warp_reduce(sum_words<A, W>(acc));
        if (lane == 0) seg_out(p, cur0, Op<A>::add(t, first));
#pragma unroll
        for (int k = 0; k < W; ++k) acc[k] = Op<A>::zero();
        // step over the segments emitted above to the one open at the row's end
        cur = cur0 + m;
        cur_start = last_pos;
        if (cur >= p.nseg) {
            cur_end = INT64_MAX;
        } else {
            const int64_t kc = cur + 1 - wb;
            if (kc < 32) {
                cur_end = __shfl_sync(0xffffffffu, win, (int)kc);
                if (kc >= 16) {  // refill the window ahead: the load overlaps the next rows
                    wb = cur + 1;
                    win = (wb + lane <= p.nseg) ? __ldg(p.offsets + wb + lane) : INT64_MAX;
                }
            } else {
                wb = cur + 1;
                win = (wb + lane <= p.nseg) ? __ldg(p.offsets + wb + lane) : INT64_MAX;
                cur_end = __shfl_sync(0xffffffffu, win, 0);
            }
        }
        if (lane == 0) acc[0] = open_end;
        return true;
    };

    // scalar chunk [c0, c1), at most 32 elements: lane l holds element c0 + l
    auto scalar_chunk = [&](int64_t c0, int64_t c1) {
        if (c0 >= c1) return;
        while (cur_end <= c0) emit_advance();
        const int64_t idx = c0 + lane;
        A one = Op<A>::zero();
        if (idx < c1) acc_elem<DT>(one, p.x, idx);
        for (;;) {
            if (idx < c1 && idx >= cur_start && idx < cur_end) acc[0] = Op<A>::add(acc[0], one);
            if (cur_end >= c1) break;
            emit_advance();
        }
    };

    // row r of vectors, words in `r_words` (lane's vector)
    auto row = [&](int64_t r, const uint32_t (&r_words)[W]) {
        const int64_t c0 = a0 + r * RW;
        const int64_t c1 = (c0 + RW < hi_al) ? c0 + RW : hi_al;
        while (cur_end <= c0) emit_advance();
        const int64_t e0 = c0 + (int64_t)lane * PV;
        const bool valid = e0 < c1;
        if (cur_end >= c1) {  // no boundary inside the row
            if (valid) {
#pragma unroll
                for (int k = 0; k < W; ++k) acc_word<DT>(acc[k], r_words[k]);
            }
            return;
        }
        if constexpr (DENSE) {
            if (row_scan(c0, c1, e0, valid, r_words)) return;
        }
        for (;;) {  // segments end inside this row (one reduction per segment)
            if (valid) {
                // element j of the lane's vector belongs to the current segment
                // when cur_start <= e0 + j < cur_end: one bit per j, from two
                // clamped offsets (static indices keep the vector in registers)
                const uint32_t m = run_mask<PV>(cur_start - e0, cur_end - e0);
#pragma unroll
                for (int j = 0; j < PV; ++j)
                    if ((m >> j) & 1u) acc_vec_elem<DT>(acc[j * W / PV], r_words, j);
            }
            if (cur_end >= c1) break;
            emit_advance();
        }
    };

    scalar_chunk(lo, a0);
    for (int64_t r = 0; r < nrows; r += UNROLL) {
        if (r > 0) {
#pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                const int64_t v = (r + u) * 32 + lane;
                if (v < nvec) ldg_vec(body + v * VB, buf[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (r + u < nrows) row(r + u, buf[u]);
    }
    scalar_chunk(hi_al, hi);
    // the segment holding the piece's last element, then any (empty) segment
    // this warp owns that starts at or after hi
    while (cur < p.nseg && cur_start < next_lo) emit_advance();

    if (p.stage == kStageTwoKernel || p.stage == kStageGridSync) {
        if (lane == 0) p.last_seg[w] = spanning;
    }
    if (p.stage == kStageGridSync) {
        cg::grid_group g = cg::this_grid();
        if (!g.is_valid()) {
            if (threadIdx.x == 0) atomicOr(p.err, 2);
            return;
        }
        g.sync();
        if (spanning >= 0) {
            const int64_t end = __ldg(p.offsets + spanning + 1);
            finish_span<A, false>(p, spanning, w, (end - 1 - base) / E, lane);
        }
    }
}

// ------------------------------------------------------- TMA form (strips)
// SR_F_BULK: the flat split with each warp's vector body streamed through its
// own ring of p.stages chunks of UNROLL rows of 32 vectors in shared memory,
// one cp.async.bulk per chunk issued by lane 0 and completing on the chunk
// stage's mbarrier (every wait bounded by p.limit_ns; on expiry the warp records
// SR_ERR_TIMEOUT, waits for the copies it issued, and stops).
//
// A chunk is cut into 32 strips, one per lane: strip t is its t-th run of
// UNROLL * VB contiguous bytes, NV 16-byte vectors.  Segment ends are resolved
// once per chunk instead of once per row or per segment:
//   - a segment inside one strip is summed by the lane that holds its end in
//     the offsets window, straight from shared memory;
//   - every lane sums its strip's vectors before the strip's first boundary
//     (head) and from its last one on (tail), the two boundary vectors split
//     element by element; one segmented scan over the lanes then closes every
//     segment that crosses a strip, and its last value is the segment open at
//     the chunk's end.
// Where every segment of a chunk is short, the strips are left out: each is
// summed by its own lane (OwnBytes, below).
//
// Resolving the ends row by row, with a warp reduction for each (as the LDG
// kernel does), bounded the ring by its instructions: it read 1M segments of 268
// BF16 values at 1.8 TB/s.  Now a chunk without an end costs 160 warp instructions, one
// with a few 460 to 510 (f32 4M x 64, bf16 1M x 268), one with 64 690 (i32 2M x 16), and
// an FP8 one with 100 2100; HBM leaves time for some 650.
// Device time before and now (~2^28 elements unless said otherwise):
//   f32   1M x 268             343 -> 179 us      f32  4M lognormal    1013 -> 190 us
//   f32   4M x 64              915 -> 191         f32  16M x 16        3110 -> 214
//   bf16  1M x 268 (0..536)    297 -> 100         fp8  100k lognormal   160 ->  60
//   i32   2^21 x 16 (0..32)    525 ->  53         bf16 4M x 39, lognormal 870 -> 108
// What bounds it now: instructions (55-70 % of the issue slots) from about five
// ends per chunk up, HBM below, and 4-7 us of search and first copies at the start.
// 80 registers, so 24 warps (two 384-thread CTAs, 1 % ahead of three of 256) are
// resident with two 4 KiB stages each: 16 warps of 112 registers took 4 % less on
// long segments and 8-12 % more on short ones.

// Sum of the elements in one 16-byte vector (four 32-bit words); compensated
// binary32 and BF16 go through PackedPairs (below) instead.
template <int DT, class A> __device__ __forceinline__ A vec_total(const uint32_t (&r)[4]) {
    if constexpr (DT == kDtI32) {
        long long s = (long long)(int)r[0];
#pragma unroll
        for (int w = 1; w < 4; ++w) asm("mad.wide.s32 %0, %1, 1, %0;" : "+l"(s) : "r"(r[w]));
        return s;
    } else if constexpr (DT == kDtFP8) {
        const float v = AccVec<kDtFP8, float, 4>::vec_sum(r);  // 16 values: exact
        if constexpr (std::is_same<A, Pair>::value) return Pair{v, 0.f};
        else return v;
    } else if constexpr (DT == kDtBF16) {
        const float a = bf16_hi_add(r[1], bf16_lo_add(r[1], bf16_hi_add(r[0], __uint_as_float(r[0] << 16))));
        const float b = bf16_hi_add(r[3], bf16_lo_add(r[3], bf16_hi_add(r[2], __uint_as_float(r[2] << 16))));
        return __fadd_rn(a, b);
    } else {
        return __fadd_rn(__fadd_rn(__uint_as_float(r[0]), __uint_as_float(r[1])),
                         __fadd_rn(__uint_as_float(r[2]), __uint_as_float(r[3])));
    }
}

// A running sum of whole vectors: the accumulator type itself, or for plain
// binary32 two partial sums in one packed register pair (PTX add.rn.f32x2:
// each half rounds like the scalar add, in half the instructions).
template <int DT, class A> struct VecPart {
    A v;
    __device__ __forceinline__ static VecPart zero() { return VecPart{Op<A>::zero()}; }
    __device__ __forceinline__ static VecPart of(const uint32_t (&r)[4]) { return VecPart{vec_total<DT, A>(r)}; }
    __device__ __forceinline__ void add(const VecPart& b) { v = Op<A>::add(v, b.v); }
    __device__ __forceinline__ A total() const { return v; }
};
template <> struct VecPart<kDtF32, float> {
    float x, y;
    __device__ __forceinline__ static VecPart zero() { return VecPart{0.f, 0.f}; }
    __device__ __forceinline__ static VecPart sum(float ax, float ay, float bx, float by) {
        VecPart t;
        asm("{ .reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
            " add.rn.f32x2 c, a, b;\n mov.b64 {%0, %1}, c; }"
            : "=f"(t.x), "=f"(t.y)
            : "f"(ax), "f"(ay), "f"(bx), "f"(by));
        return t;
    }
    __device__ __forceinline__ static VecPart of(const uint32_t (&r)[4]) {
        return sum(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]), __uint_as_float(r[3]));
    }
    __device__ __forceinline__ void add(const VecPart& b) { *this = sum(x, y, b.x, b.y); }
    __device__ __forceinline__ float total() const { return __fadd_rn(x, y); }
};

// Compensated binary32 and BF16: two (sum, correction) pairs in packed registers.
// Each TwoSum (Knuth's, each half rounded like the scalar form) takes six packed
// instructions for two pairs: a vector costs 14 (f32) or 28 (BF16) instead of 28 or 56.
__device__ __forceinline__ void two_sum_packed(float ax, float ay, float bx, float by, float& sx, float& sy,
                                               float& ex, float& ey) {
    asm("{ .reg .b64 a, b, t, bp, ap, d1, d2, e;\n"
        " mov.b64 a, {%4, %5};\n mov.b64 b, {%6, %7};\n"
        " add.rn.f32x2 t, a, b;\n sub.rn.f32x2 bp, t, a;\n sub.rn.f32x2 ap, t, bp;\n"
        " sub.rn.f32x2 d1, a, ap;\n sub.rn.f32x2 d2, b, bp;\n add.rn.f32x2 e, d1, d2;\n"
        " mov.b64 {%0, %1}, t;\n mov.b64 {%2, %3}, e; }"
        : "=f"(sx), "=f"(sy), "=f"(ex), "=f"(ey)
        : "f"(ax), "f"(ay), "f"(bx), "f"(by));
}
struct PackedPairs {
    float sx, sy, cx, cy;
    __device__ __forceinline__ static PackedPairs zero() { return PackedPairs{0.f, 0.f, 0.f, 0.f}; }
    __device__ __forceinline__ static PackedPairs of_sum(float ax, float ay, float bx, float by) {
        PackedPairs t;
        two_sum_packed(ax, ay, bx, by, t.sx, t.sy, t.cx, t.cy);
        return t;
    }
    __device__ __forceinline__ void add(const PackedPairs& b) {
        float ex, ey;
        two_sum_packed(sx, sy, b.sx, b.sy, sx, sy, ex, ey);
        VecPart<kDtF32, float> c = VecPart<kDtF32, float>::sum(cx, cy, b.cx, b.cy);
        c = VecPart<kDtF32, float>::sum(c.x, c.y, ex, ey);
        cx = c.x;
        cy = c.y;
    }
    __device__ __forceinline__ Pair total() const { return Op<Pair>::add(Pair{sx, cx}, Pair{sy, cy}); }
};
template <> struct VecPart<kDtF32, Pair> : PackedPairs {
    __device__ __forceinline__ static VecPart zero() { return VecPart{PackedPairs::zero()}; }
    __device__ __forceinline__ static VecPart of(const uint32_t (&r)[4]) {
        return VecPart{of_sum(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]),
                              __uint_as_float(r[3]))};
    }
};
template <> struct VecPart<kDtBF16, Pair> : PackedPairs {
    __device__ __forceinline__ static VecPart zero() { return VecPart{PackedPairs::zero()}; }
    __device__ __forceinline__ static PackedPairs two_words(uint32_t a, uint32_t b) {
        return of_sum(__uint_as_float(a << 16), __uint_as_float(b << 16), __uint_as_float(a & 0xffff0000u),
                      __uint_as_float(b & 0xffff0000u));
    }
    __device__ __forceinline__ static VecPart of(const uint32_t (&r)[4]) {
        PackedPairs t = two_words(r[0], r[1]);
        t.add(two_words(r[2], r[3]));
        return VecPart{t};
    }
};

// The low n bits (n <= 0: none, n >= 32: all).
__device__ __forceinline__ uint32_t low_bits(int n) {
    uint32_t above;  // PTX shl: 0 from 32 on
    asm("shl.b32 %0, %1, %2;" : "=r"(above) : "r"(0xffffffffu), "r"(max(n, 0)));
    return ~above;
}
// Zero the elements of a vector at or after index n (keep_below) or before it
// (keep_from); 0 <= n <= 16 / EB.  A zeroed word is +0 in every input type.
template <int EB> __device__ __forceinline__ void keep_below(uint32_t (&r)[4], int n) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        if constexpr (EB == 4) r[w] = w < n ? r[w] : 0u;
        else r[w] &= low_bits(8 * EB * n - 32 * w);
    }
}
template <int EB> __device__ __forceinline__ void keep_from(uint32_t (&r)[4], int n) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        if constexpr (EB == 4) r[w] = w >= n ? r[w] : 0u;
        else r[w] &= ~low_bits(8 * EB * n - 32 * w);
    }
}

// A warp's piece, e elements of `eb` bytes in an even split, as large as it has to be for
// chunks of `ce` (sr_segparams.h).  From three quarters of a chunk on the even split stays:
// fewer warps then save nothing (4096 segments of 775 f32: 10.2 us, 10.0).
__device__ __forceinline__ int64_t strip_piece(int64_t e, int64_t n, int64_t nseg, int ce, int eb) {
    if (n * eb >= (int64_t)kLongMean * nseg) return e < ce / 4 * 3 ? ce : e;
    return e < ce / kPieceParts ? ce / kPieceParts : e;
}

// Offsets fetched into L2 this far ahead of the window: the one after `nxt`.  Further
// ahead they are more often gone again (16M x 16 f32: 211 us with 64, 216 with 192,
// 231 with 256).
constexpr int kAheadOffsets = 64;
// Longest segment (bytes) one lane sums alone, about where that costs a chunk
// as many instructions as the strips do.
template <int DT> struct OwnBytes { static constexpr int v = 256; };
template <> struct OwnBytes<kDtI32> { static constexpr int v = 192; };
template <> struct OwnBytes<kDtBF16> { static constexpr int v = 192; };
template <> struct OwnBytes<kDtFP8> { static constexpr int v = 128; };

// Runs of empty segments (padded offsets, keys that never occur) lie at one element, so the
// split by elements leaves a whole run to one warp: a million segments of 16 with three
// million empty ones behind them took 560 ms, one step each.  Now (32 us without the run):
// 36 us with it behind or before the data, 41 in the middle.
//   - The blocks of kEmptyBlock segments that are all empty are zeroed by all warps in turn
//     (two loads per block, beside the kernel's first ones).
//   - The warp that comes upon a run where a chunk or the piece starts or ends looks for the
//     run's end and writes what lies outside those blocks (skip_empty).
//   - A chunk takes the ends inside it a window of 32 at a time, 0.4 us each.  A piece with
//     more than kFewSegments + 1/16 of its elements is therefore searched for runs of kRun
//     entries and walked in stretches that end at them (next_run).  Fewer cost less than
//     the looking: with 1/32, 16M segments of 16 lost another 1.5 %.
// To look at every window instead costs 5-10 % on short segments: 4 instructions, but 60
// more a chunk for registers that the strips then lack.
constexpr int kEmptyBlock = 1024, kFewSegments = 1024, kRun = 512;

// Zero out[a], ..., out[b - 1], `es` bytes each (4 or 8); whole warp calls.
__device__ __forceinline__ void zero_out(void* out, int es, int64_t a, int64_t b, int lane) {
    uint32_t* o = reinterpret_cast<uint32_t*>(out);
    const int64_t hi = b * (es / 4);
    for (int64_t i = a * (es / 4) + lane; i < hi; i += 32) o[i] = 0u;
}
// The window of offsets a warp of the strip kernel walks: lane k holds offsets[wb + k]
// in win and offsets[wb + 32 + k] in nxt (INT64_MAX past the last).
struct SegWindow {
    int64_t wb, win, nxt;
    int kb;  // entry of the open segment's end
};
__device__ __forceinline__ int64_t offset_at(const int64_t* off, int64_t nseg, int64_t i) {
    return i <= nseg ? __ldg(off + i) : INT64_MAX;
}

// Closes the empty segments at element `at`, where the open segment starts (beyond two
// windows, only those outside the blocks that are all empty), and opens the one after them.
// Whole warp calls; out of line, or its registers would be taken from the strips (inlined:
// 16M x 16 2-5 % slower).
static __device__ __noinline__ SegWindow skip_empty(const int64_t* off, int64_t nseg, void* out, int es, int64_t at,
                                                    SegWindow w) {
    const int lane = threadIdx.x & 31;
    for (;;) {
        const int cnt = __popc(__ballot_sync(0xffffffffu, lane >= w.kb && w.win == at));
        zero_out(out, es, w.wb + w.kb - 1, w.wb + w.kb - 1 + cnt, lane);
        w.kb += cnt;
        if (w.kb < 32) return w;
        if (!__all_sync(0xffffffffu, w.nxt == at)) {
            w.win = w.nxt;
            w.wb += 32;
        } else {
            // lo: the first index with offsets[lo] > at (nseg + 1: none), looked for at
            // power-of-two distances, then in 32 equal parts at a time
            int64_t lo = w.wb + 64, hi = nseg + 1;
            {
                const int64_t k = lo + ((int64_t)1 << lane) - 1;
                const unsigned m = __ballot_sync(0xffffffffu, k >= hi || __ldg(off + k) > at);
                const int b = m ? __ffs(m) - 1 : 32;
                if (b < 32) hi = min(hi, lo + ((int64_t)1 << b) - 1);
                if (b > 0) lo += (int64_t)1 << (b - 1);
            }
            while (lo < hi) {
                const int64_t step = (hi - lo + 31) / 32;
                const int64_t k = lo + lane * step;
                const unsigned m = __ballot_sync(0xffffffffu, k >= hi || __ldg(off + k) > at);
                const int b = m ? __ffs(m) - 1 : 32;
                if (b < 32) hi = min(hi, lo + b * step);
                if (b > 0) lo += (b - 1) * step + 1;
            }
            // segments s0 .. end - 1 are empty too
            const int64_t s0 = w.wb + 31, end = lo - 1;
            const int64_t b0 = (s0 + kEmptyBlock - 1) / kEmptyBlock * kEmptyBlock, b1 = end / kEmptyBlock * kEmptyBlock;
            zero_out(out, es, s0, min(end, b0), lane);
            zero_out(out, es, max(b0, b1), end, lane);
            w.wb = lo;
            w.win = offset_at(off, nseg, lo + lane);
        }
        w.kb = 0;
        w.nxt = offset_at(off, nseg, w.wb + 32 + lane);
    }
}

// The element at which the first run of empty segments that takes kRun entries from entry i
// of the offsets on (i + k kRun to i + k kRun + kRun) starts, before element `hi`; hi if
// there is none (whole warp calls).
static __device__ __noinline__ int64_t next_run(const int64_t* off, int64_t nseg, int64_t i, int64_t hi) {
    const int lane = threadIdx.x & 31;
    for (;; i += 32 * kRun) {
        const int64_t a = offset_at(off, nseg, i + kRun * lane), b = offset_at(off, nseg, i + kRun * (lane + 1));
        const unsigned m = __ballot_sync(0xffffffffu, a == b || b >= hi);
        if (m != 0u) return min(hi, __shfl_sync(0xffffffffu, a == b ? a : hi, __ffs(m) - 1));
    }
}

template <int DT, bool COMP, int VB, int UNROLL>
__global__ void __maxnreg__(80) seg_strip_kernel(const SegParams p) {
    using A = typename Acc<DT, COMP>::T;
    using VP = VecPart<DT, A>;
    constexpr int EB = SegElem<DT>::v;
    constexpr int PV = VB / EB;                             // elements per vector of the flat split
    constexpr uint32_t CHUNK = (uint32_t)UNROLL * 32u * VB;  // bytes of one ring stage
    constexpr int CE = (int)CHUNK / EB;                     // elements of a chunk
    constexpr int SE = CE / 32;                             // elements of a strip (a power of two)
    constexpr int EV = 16 / EB;                             // elements of a 16-byte vector
    constexpr int NV = SE / EV;                             // 16-byte vectors of a strip
    constexpr int kOwn = OwnBytes<DT>::v / EB;
    // FP8 and compensated BF16 vectors take 40 to 50 instructions each: with their
    // loops unrolled the warps wait for instructions (FP8: 72 us against 63 on
    // 100,000 lognormal segments of 2^28 elements)
    constexpr bool kCompact = DT == kDtFP8 || (COMP && DT == kDtBF16);
    constexpr int UN = kCompact && NV > 2 ? 2 : NV;
    grid_dependency_wait();
    allow_dependents();
    if (p.bad != nullptr && __ldcg(p.bad) != 0) return;  // offsets failed the check: read nothing
    const int lane = threadIdx.x & 31;
    const int w = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // at most 65536 warps
    const int Wn = (int)(gridDim.x * blockDim.x) >> 5;
    const int64_t base = __ldg(p.offsets);
    const int64_t N = __ldg(p.offsets + p.nseg) - base;
    int64_t E = (N + Wn - 1) / Wn;
    E = ((E + PV - 1) / PV) * PV;
    E = strip_piece(E, N, p.nseg, CE, EB);
    const int64_t lo = base + (w * E < N ? w * E : N);
    const int64_t hi = base + ((w + 1) * E < N ? (w + 1) * E : N);

    // A stretch [from, to) of the piece (all of it, unless there are long runs of empty
    // segments): scalar head, vector body of `left` chunks (last_ce elements in the last),
    // scalar tail.
    int head, left, last_ce, tail;
    auto geometry = [&](int64_t from, int64_t to) {
        const uintptr_t addr = reinterpret_cast<uintptr_t>(p.x) + (uintptr_t)from * EB;
        head = (int)(((uintptr_t)VB - addr % VB) % VB) / EB;
        if (head > to - from) head = (int)(to - from);
        const int64_t body = (to - from - head) / PV * PV;
        left = (int)((body + CE - 1) / CE);
        last_ce = (int)(body - (int64_t)(left - 1) * CE);
        tail = (int)(to - from - head - body);
    };
    geometry(lo, hi);
    // segments that start at hi are this warp's too (elsewhere they are the next one's)
    const int64_t last = w == Wn - 1 || base + (w + 1) * E > hi;
    // base, E, hi and last are wanted only where a segment crosses the piece's ends or a
    // stretch ends: the lanes keep a word each of them
    const uint32_t stash = (uint32_t)((lane & 4 ? (lane & 2 ? last : hi) : lane & 2 ? E : base) >> (lane & 1 ? 32 : 0));
    auto stashed = [&](int at) {
        return (int64_t)((uint64_t)__shfl_sync(0xffffffffu, stash, at) |
                         (uint64_t)__shfl_sync(0xffffffffu, stash, at + 1) << 32);
    };

    extern __shared__ __align__(1024) unsigned char seg_dsm[];
    const int wib = threadIdx.x >> 5, nwib = blockDim.x >> 5, S = p.stages;
    const uint32_t ring = smem_u32(seg_dsm) + (uint32_t)(wib * S) * CHUNK;
    const uint32_t bars = smem_u32(seg_dsm) + (uint32_t)(nwib * S) * CHUNK + (uint32_t)(wib * S) * 8u;
    // the strip table: word t describes strip t's boundaries of one offsets window
    const uint32_t table =
        smem_u32(seg_dsm) + (uint32_t)(nwib * S) * (CHUNK + 8u) + (uint32_t)(wib * kStripTableBytes);
    // lane 0: copy the chunk at src, of l up to the last one, into ring stage st, if there is one
    auto issue = [&](const unsigned char* src, int l, int st) {
        if (l <= 0) return;
        const uint32_t bytes = l == 1 ? (uint32_t)last_ce * EB : CHUNK;
        mbar_arrive_expect_tx(bars + 8u * st, bytes);
        bulk_g2s(ring + (uint32_t)st * CHUNK, src, bytes, bars + 8u * st);
    };
    // the ring's first copies (24 warps' rings are 30 MB for the chip: issued before
    // the search they held the searching warps up to 8 us, now 4)
    int64_t wb, win, far;
    auto fill = [&]() {
        far = offset_at(p.offsets, p.nseg, wb + kFewSegments + E / 16);
        if (lane == 0) {
            for (int j = 0; j < S; ++j) mbar_init(bars + 8u * j, 1);
            mbar_fence_init();
            for (int j = 0; j < S; ++j) issue(p.x + (lo + head + (int64_t)j * CE) * EB, left - j, j);
        }
        __syncwarp();
    };

    // this lane's block of segments, all empty if its first and last offset are equal
    const int64_t nblk = p.nseg / kEmptyBlock;
    int64_t blk = w + (int64_t)lane * Wn, blk0 = 0, blk1 = 1;
    if (blk < nblk) {
        blk0 = __ldg(p.offsets + blk * kEmptyBlock);
        blk1 = __ldg(p.offsets + (blk + 1) * kEmptyBlock);
    }

    // Stream state (warp-uniform).  The offsets window: lane k holds
    // offsets[wb + k] in win and offsets[wb + 32 + k] in nxt (loaded one window
    // ahead).  Entry kb is the end of the open segment, wb + kb - 1.
    const int64_t at = N > 0 ? (int64_t)((float)(w * E) / (float)N * (float)p.nseg) : 0;
    int r0 = 0;
    if (w * E <= N) {
        r0 = (int)(warp_search(p.offsets, p.nseg, base + w * E, at < p.nseg ? at : p.nseg, lane, wb, win, fill) - wb);
    } else {  // nothing for this warp: past the last segment
        wb = p.nseg;
        win = far = INT64_MAX;
    }
    int64_t nxt = (wb + 32 + lane <= p.nseg) ? __ldg(p.offsets + wb + 32 + lane) : INT64_MAX;
    // the open segment began in an earlier warp's piece
    bool cont = lo < hi && __shfl_sync(0xffffffffu, win, r0) > lo;
    int kb = cont ? r0 : r0 + 1;
    int64_t cur_end = __shfl_sync(0xffffffffu, win, kb);
    // This lane's part of the open segment: one addition per chunk, 72 in a warp's piece
    // of 2^28 binary32 elements (in a plain chain, constant data came out 5.6 eps32 off
    // in 4200 segments of 60,000 where 4 is the gate).
    RunSum<A> acc = RunSum<A>::of(Op<A>::zero());
    bool spread = false;  // acc is nonzero in lanes other than lane 0

    while (w < nblk) {  // blocks of empty segments
        unsigned m = __ballot_sync(0xffffffffu, blk0 == blk1);
        for (; m != 0u; m &= m - 1u) {
            const int64_t b = __shfl_sync(0xffffffffu, blk, __ffs(m) - 1);
            zero_out(p.out, std::is_same<A, long long>::value || p.fp64 ? 8 : 4, b * kEmptyBlock, (b + 1) * kEmptyBlock,
                     lane);
        }
        blk += 32 * (int64_t)Wn;
        if (__all_sync(0xffffffffu, blk >= nblk)) break;
        blk0 = blk < nblk ? __ldg(p.offsets + blk * kEmptyBlock) : 0;
        blk1 = blk < nblk ? __ldg(p.offsets + (blk + 1) * kEmptyBlock) : 1;
    }

    auto next_window = [&]() {
        win = nxt;
        wb += 32;
        kb = 0;
        nxt = (wb + 32 + lane <= p.nseg) ? __ldg(p.offsets + wb + 32 + lane) : INT64_MAX;
        if (wb + kAheadOffsets + lane <= p.nseg)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.offsets + wb + kAheadOffsets + lane));
    };
    // this warp's piece of segment s, owned by an earlier warp; v in lane 0
    auto emit_first = [&](int64_t s, A v) {
        cont = false;
        if (p.stage == kStageAtomic) {
            if (lane == 0) seg_atomic(p, s, v);
            return;
        }
        if (lane == 0) carry_store(p, p.carry_first, w, v);
        if (p.stage == kStageLastBlock) {
            const int64_t b = stashed(0), e = stashed(2);
            span_arrive<A, true>(p, s, (__ldg(p.offsets + s) - b) / e, (__ldg(p.offsets + s + 1) - 1 - b) / e, lane);
        }
    };
    // the open segment's sum so far, in lane 0; acc restarts at zero
    auto take_acc = [&]() {
        const A v = spread ? warp_reduce(acc.total()) : acc.only();
        acc = RunSum<A>::of(Op<A>::zero());
        spread = false;
        return v;
    };
    // close the open segment (it ends inside the piece) and move to the next one
    auto emit_advance = [&]() {
        const A v = take_acc();
        if (cont) emit_first(wb + kb - 1, v);
        else if (lane == 0) seg_out(p, wb + kb - 1, v);
        if (++kb == 32) next_window();
        cur_end = __shfl_sync(0xffffffffu, win, kb);
    };
    auto skip = [&](int64_t at) {  // skip_empty on the stream state
        const int es = std::is_same<A, long long>::value || p.fp64 ? 8 : 4;
        const SegWindow n = skip_empty(p.offsets, p.nseg, p.out, es, at, SegWindow{wb, win, nxt, kb});
        wb = n.wb;
        win = n.win;
        nxt = n.nxt;
        kb = n.kb;
    };

    // Lane l reads vector j ^ sw of its strip at step j: eight consecutive lanes
    // then hit eight different 16-byte bank groups (strips are a multiple of 32
    // bytes apart, which in order is an up to 8-way conflict).
    const int sw = (NV >= 8 ? lane : lane / (8 / NV)) & (NV - 1);

    // elements [a, b) of the chunk in stage sb, a < b, summed by one lane, which
    // starts at a vector of its own choosing (with equal lengths of a power of two
    // the first ones would all lie on the same banks)
    auto own_sum = [&](uint32_t sb, int a, int b) {
        const uint32_t va = (unsigned)a / EV, vb = (unsigned)(b - 1) / EV;
        const int nb = b - (int)vb * EV;  // elements of the last vector
        uint32_t r[4];
        if constexpr (DT == kDtFP8) {
            // one copy of the code: the first vector, the last, then those between, so
            // that all lanes mask in the same two steps (masked wherever a lane's turn
            // came, nearly every step did: 1.5M segments of 41 49.2 -> 46.4 us, 4M of 64 78.8 -> 74.2)
            uint32_t i = va, next = va + 1u + ((uint32_t)lane & 7u);
            if (next >= vb) next = va + 1u;
            VP v = VP::zero();
#pragma unroll 1
            for (uint32_t k = 0; k <= vb - va; ++k) {
                lds_vec(sb + 16u * i, r);
                if (k < 2) {
                    if (k == 0) keep_from<EB>(r, a & (EV - 1));
                    if (i == vb) keep_below<EB>(r, nb);
                }
                v.add(VP::of(r));
                if (k == 0) {
                    i = vb;
                } else {
                    i = next;
                    if (++next >= vb) next = va + 1u;
                }
            }
            return v.total();
        } else {  // the masked ends apart from the whole vectors between them
            lds_vec(sb + 16u * va, r);
            keep_from<EB>(r, a & (EV - 1));
            if (va == vb) keep_below<EB>(r, nb);
            VP v = VP::of(r);
            if (va != vb) {
                const uint32_t m = vb - va - 1;
                uint32_t i = (uint32_t)lane & 7u;
                if (i >= m) i = 0;
                for (uint32_t n = 0; n < m; ++n) {
                    lds_vec(sb + 16u * (va + 1u + i), r);
                    v.add(VP::of(r));
                    if (++i == m) i = 0;
                }
                lds_vec(sb + 16u * vb, r);
                keep_below<EB>(r, nb);
                v.add(VP::of(r));
            }
            return v.total();
        }
    };

    // the chunk of `ce` elements from c0 in ring stage `sb`, zero-filled to CHUNK bytes
    auto chunk = [&](const int64_t c0, int ce, uint32_t sb) {
        const uint32_t strip = sb + (uint32_t)lane * (CHUNK / 32u);
        const uint32_t v0 = strip + 16u * (uint32_t)sw;  // the strip is aligned to its size
        if (cur_end >= c0 + ce) {  // no segment ends inside the chunk
            VP v[2] = {VP::zero(), VP::zero()};
#pragma unroll (UN / 2)
            for (int j = 0; j < NV; j += 2) {
                uint32_t r0[4], r1[4];
                lds_vec(v0 ^ (16u * j), r0);
                lds_vec(v0 ^ (16u * j + 16u), r1);
                v[0].add(VP::of(r0));
                v[1].add(VP::of(r1));
            }
            v[0].add(v[1]);
            acc.add(v[0].total());
            spread = true;
            return;
        }
        // Boundaries of the chunk, one offsets window at a time; positions
        // relative to c0.  prev: the boundary before the window's first, -1 when
        // the open segment began at c0 or before.
        int prev = -1, rp, rpp;
        bool is_b, short_only;
        auto window = [&]() {
            const int64_t ahead = win - c0;
            rp = ahead < ce ? (int)ahead : 2 * CE;
            is_b = lane >= kb && rp < ce;
            rpp = __shfl_up_sync(0xffffffffu, rp, 1);  // the boundary before this lane's
            if (lane == kb) rpp = prev;
        };
        // steps past the window's boundaries; true when more of the chunk's follow
        auto advance = [&]() {
            kb += __popc(__ballot_sync(0xffffffffu, is_b));
            prev = __shfl_sync(0xffffffffu, rp, kb - 1);
            if (kb < 32) return false;
            next_window();
            return __shfl_sync(0xffffffffu, win, 0) < c0 + ce;
        };
        // windows whose segments are all short: every lane sums the one that ends
        // at its boundary, straight from shared memory
        window();
        short_only = true;
        const int last = __shfl_sync(0xffffffffu, rp, 31);
        if (last < ce) {  // the window after this one has a say too: mixing both ways in one chunk costs both
            const int64_t ahead = nxt - c0;
            const int np = ahead < ce ? (int)ahead : 2 * CE;
            int npp = __shfl_up_sync(0xffffffffu, np, 1);
            if (lane == 0) npp = last;
            short_only = !__any_sync(0xffffffffu, np < ce && np - npp > kOwn);
        }
        while (short_only) {
            const int from = rpp > 0 ? rpp : 0;
            if (__any_sync(0xffffffffu, is_b && rp - from > kOwn)) break;
            A v = Op<A>::zero();
            if (is_b && rp > from) v = own_sum(sb, from, rp);
            bool write = is_b;
            if (prev < 0) {  // the first one: with what earlier chunks hold of it
                const A before = Op<A>::shfl(take_acc(), 0);
                if (lane == kb) v = Op<A>::add(before, v);
                if (cont) {
                    write = is_b && lane != kb;
                    emit_first(wb + kb - 1, Op<A>::shfl(v, kb));
                }
            }
            if (write) seg_out(p, wb + lane - 1, v);
            if (advance()) {
                window();
                continue;
            }
            // the segment open at the chunk's end: [prev, CE), vectors spread over the lanes
            VP t = VP::zero();
            for (uint32_t k = (unsigned)prev / EV + lane; k < 32u * NV; k += 32u) {
                uint32_t r[4];
                lds_vec(sb + 16u * k, r);
                if (k == (unsigned)prev / EV) keep_from<EB>(r, prev & (EV - 1));
                t.add(VP::of(r));
            }
            acc = RunSum<A>::of(t.total());
            spread = true;
            cur_end = __shfl_sync(0xffffffffu, win, kb);
            return;
        }
        // the rest of the chunk by strips
        const int begin = prev;  // >= 0: a boundary whose segment is closed already
        int qf = SE, ql = SE;    // this lane's strip: first and last boundary (SE: none)
        int64_t qseg = 0;        // the segment that ends at the first one
        for (;;) {
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(table + 4u * lane), "r"(0xffffffffu) : "memory");
            __syncwarp();
            const int rpn = __shfl_down_sync(0xffffffffu, rp, 1);  // the boundary after this lane's
            if (is_b) {
                const int t = (int)((unsigned)rp / SE), q = (int)((unsigned)rp % SE);
                if (rpp >= t * SE) {  // starts and ends inside strip t
                    seg_out(p, wb + lane - 1, rp > rpp ? own_sum(sb, rpp, rp) : Op<A>::zero());
                } else {  // the strip's first boundary
                    const unsigned short e = (unsigned short)(q | (lane << 8));
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(table + 4u * t), "h"(e) : "memory");
                }
                // the strip's last boundary in this window (a later window may hold one after it)
                if (lane == 31 || rpn >= (t + 1) * SE) {
                    const unsigned short e = (unsigned short)q;
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(table + 4u * t + 2u), "h"(e) : "memory");
                }
            }
            __syncwarp();
            uint32_t e;
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(e) : "r"(table + 4u * lane) : "memory");
            if ((e & 0xffffu) != 0xffffu) {
                qf = (int)(e & 0xffu);
                qseg = wb + (int)((e >> 8) & 0xffu) - 1;
            }
            if ((e >> 16) != 0xffffu) ql = (int)(e >> 16);
            if (!advance()) break;
            window();
        }
        cur_end = __shfl_sync(0xffffffffu, win, kb);

        bool closes = qf < SE;
        if (begin >= 0 && lane == (int)((unsigned)begin / SE)) {
            qf = begin & (SE - 1);  // the run from here on is new, and nothing is left to close
            if (ql == SE) ql = qf;
            closes = false;
        }
        const bool has_b = qf < SE;
        const unsigned tmask = __ballot_sync(0xffffffffu, has_b);
        const int vf = (int)((unsigned)qf / EV), vl = (int)((unsigned)ql / EV);  // NV when there is none
        VP hv = VP::zero(), tv = VP::zero();
#pragma unroll (UN)
        for (int j = 0; j < NV; ++j) {
            const int kv = j ^ sw;
            uint32_t r[4];
            lds_vec(v0 ^ (16u * j), r);
            const VP v = VP::of(r);
            if (kv < vf) hv.add(v);
            if (kv > vl) tv.add(v);
        }
        if (has_b) {  // the boundary vectors
            uint32_t r[4];
            lds_vec(strip + 16u * vf, r);
            keep_below<EB>(r, qf & (EV - 1));
            hv.add(VP::of(r));
            lds_vec(strip + 16u * vl, r);
            keep_from<EB>(r, ql & (EV - 1));
            tv.add(VP::of(r));
        }
        const A head = hv.total();
        // segmented inclusive scan of the open runs over the strips: before the
        // step with distance d a lane's partial covers lanes [lane - d + 1,
        // lane], and takes in the lanes before them unless one of its own holds
        // a boundary, that is while d <= reach
        const unsigned upto = tmask & ((2u << lane) - 1u);  // boundary lanes 0 .. lane (2 << 31 wraps to 0)
        const int reach = upto ? lane - (31 - __clz(upto)) : lane;
        A x = has_b ? tv.total() : head;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const A xo = Op<A>::shfl_up(x, d);
            if (d <= reach) x = Op<A>::add(xo, x);
        }
        A closed = Op<A>::shfl_up(x, 1);  // the run open at the end of the strip before
        closed = lane == 0 ? head : Op<A>::add(closed, head);
        const A open_end = Op<A>::shfl(x, 31);
        // the open segment of the chunks before is the first to end: its sum is rounded
        // once here (entering at strip 0 it was rounded at every step of the scan)
        const int fl = __ffs(tmask) - 1;
        const A before = Op<A>::shfl(take_acc(), 0);
        if (lane == fl) closed = Op<A>::add(before, closed);
        if (lane == 0) acc = RunSum<A>::of(open_end);
        if (cont) {  // it began in an earlier warp's piece
            emit_first(__shfl_sync(0xffffffffu, qseg, fl), Op<A>::shfl(closed, fl));
            closes = closes && lane != fl;
        }
        if (closes) seg_out(p, qseg, closed);
    };

    // The walk: of each stretch the head's elements, the chunks, the tail's elements;
    // everything before `pos` is summed.  One loop, so that the code which closes segments
    // is there once.
    int st = 0;
    uint32_t par = 0;
    bool bail = false;
    int flight = left < S ? left : S;  // copies under way when a wait expires
    int64_t pos = lo;
    // Many segments: long runs of empty ones may be among them, which a chunk would take a
    // window at a time.  The piece is then walked in stretches that end where one starts.
    bool more = far < hi && next_run(p.offsets, p.nseg, wb + kb, hi) < hi;
    if (__builtin_expect(more, 0)) {
        for (; flight > 0; --flight) {
            bail = !__all_sync(0xffffffffu, mbar_wait_bounded(bars + 8u * st, par, p.limit_ns));
            if (bail) break;
            if (++st == S) {
                st = 0;
                par ^= 1u;
            }
        }
        head = left = tail = 0;
    }
    while (!bail) {
        const bool end = head + left + tail == 0;
        while (__builtin_expect(cur_end <= pos, 0)) {  // segments that end here
            emit_advance();
            if (end && !more && !stashed(6)) {
                wb = p.nseg;  // nothing open: past the last segment
                kb = 1;
                break;
            }
            if (cur_end == pos) {
                skip(pos);
                cur_end = __shfl_sync(0xffffffffu, win, kb);
            }
        }
        if (__builtin_expect(end, 0)) {
            if (!more) break;
            const int64_t to = next_run(p.offsets, p.nseg, wb + kb, stashed(4));
            more = to < stashed(4);
            geometry(pos, to);
            if (lane == 0) {
                fence_proxy_async_smem();
                for (int j = 0; j < S; ++j)
                    issue(p.x + (pos + head + (int64_t)j * CE) * EB, left - j, st + j < S ? st + j : st + j - S);
            }
            __syncwarp();
            continue;
        }
        if (__builtin_expect(head > 0 || left == 0, 0)) {  // elements, at most 32, up to the open segment's end
            int n = head > 0 ? head : tail;
            if (cur_end - pos < n) n = (int)(cur_end - pos);
            if (lane < n) {
                A one = Op<A>::zero();
                acc_elem<DT>(one, p.x, pos + lane);
                acc.add(one);
            }
            spread = true;
            if (head > 0) head -= n;
            else tail -= n;
            pos += n;
            continue;
        }
        do {  // chunks, until a segment ends where one starts
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(bars + 8u * st, par, p.limit_ns))) {
                flight = left < S ? left : S;
                bail = true;
                break;
            }
            const int ce = left == 1 ? last_ce : CE;
            const uint32_t sb = ring + (uint32_t)st * CHUNK;
            if (ce < CE) {  // a short copy (the piece's last): zeros behind it
                for (uint32_t b = (uint32_t)ce * EB + 16u * lane; b < CHUNK; b += 512u)
                    asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(sb + b), "r"(0) : "memory");
                __syncwarp();
            }
            chunk(pos, ce, sb);
            __syncwarp();  // every lane has read the stage
            if (lane == 0) {
                fence_proxy_async_smem();
                issue(p.x + (pos + (int64_t)S * CE) * EB, left - S, st);
            }
            pos += ce;
            --left;
            if (++st == S) {
                st = 0;
                par ^= 1u;
            }
        } while (left > 0 && cur_end > pos);
    }
    if (bail && lane == 0) {
        atomicOr(p.err, kErrTimeout);
        // leave no copy writing this CTA's shared memory: wait for the ones under way,
        // bounded separately (>= 1 s)
        const uint64_t drain = p.limit_ns > 1000000000ull ? p.limit_ns : 1000000000ull;
        for (; flight > 0; --flight) {
            mbar_wait_bounded(bars + 8u * st, par, drain);
            if (++st == S) {
                st = 0;
                par ^= 1u;
            }
        }
    }
    int64_t spanning = -1;  // the owned segment that runs past this piece
    if (!bail) {            // a timeout's results are void (SR_ERR_TIMEOUT): nothing left to finish
        if (cont) {  // the whole piece lies inside an earlier warp's segment
            emit_first(wb + kb - 1, take_acc());
        } else if (wb + kb <= p.nseg) {
            spanning = wb + kb - 1;
            const A v = take_acc();
            if (p.stage == kStageAtomic) {
                if (lane == 0) seg_atomic(p, spanning, v);
            } else {
                if (lane == 0) carry_store(p, p.carry_last, w, v);
                if (p.stage == kStageLastBlock)
                    span_arrive<A, true>(p, spanning, w, (cur_end - 1 - stashed(0)) / stashed(2), lane);
            }
        }
    }

    if (p.stage == kStageTwoKernel || p.stage == kStageGridSync) {
        if (lane == 0) p.last_seg[w] = spanning;
    }
    if (p.stage == kStageGridSync) {
        cg::grid_group g = cg::this_grid();
        if (!g.is_valid()) {
            if (threadIdx.x == 0) atomicOr(p.err, 2);
            return;
        }
        g.sync();
        if (spanning >= 0) {
            const int64_t end = __ldg(p.offsets + spanning + 1);
            finish_span<A, true>(p, spanning, w, (end - 1 - stashed(0)) / stashed(2), lane);
        }
    }
}

// Second kernel of the two-kernel form: one warp per first-kernel warp.
template <int DT, bool COMP>
__global__ void __launch_bounds__(256) seg_finish_kernel(const SegParams p, int64_t Wn, int PV, int chunk,
                                                          int late) {
    using A = typename Acc<DT, COMP>::T;
    grid_dependency_wait();  // the implicit barrier: every first-kernel warp has finished
    // The next call's first kernel is let in at once, but (late) at the end where its CTAs
    // are three to an SM: while these here hold an SM they come in unevenly (4M lognormal
    // segments, strip kernel of 256 threads: 221 us a call, 189; two to an SM: no change).
    if (!late) allow_dependents();
    if (p.bad != nullptr && __ldcg(p.bad) != 0) return;
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= Wn) return;
    const int64_t s = __ldcg(p.last_seg + w);
    if (s < 0) return;
    const int64_t base = __ldg(p.offsets);
    const int64_t N = __ldg(p.offsets + p.nseg) - base;
    int64_t E = (N + Wn - 1) / Wn;  // the first kernel's piece size
    E = ((E + PV - 1) / PV) * PV;
    if (E < PV) E = PV;
    if (chunk) E = strip_piece(E, N, p.nseg, chunk, SegElem<DT>::v);
    const int64_t end = __ldg(p.offsets + s + 1);
    finish_span<A, true>(p, s, w, (end - 1 - base) / E, lane);
}

// The dense variant exists for at most 4 rows in flight per warp: with 8 its
// larger state through the hot loop cost 20-65 % on sparse layouts.
template <int DT, bool COMP, int VB, bool DENSE>
inline const void* pick_seg(int unroll) {
    switch (unroll) {
    case 1: return (const void*)seg_kernel<DT, COMP, VB, 1, DENSE>;
    case 2: return (const void*)seg_kernel<DT, COMP, VB, 2, DENSE>;
    case 4: return (const void*)seg_kernel<DT, COMP, VB, 4, DENSE>;
    case 8: return DENSE ? nullptr : (const void*)seg_kernel<DT, COMP, VB, 8, false>;
    default: return nullptr;
    }
}
// The TMA form: chunks of 2, 4 or 8 rows, no dense pass.
template <int DT, bool COMP, int VB>
inline const void* pick_seg_bulk(int unroll) {
    switch (unroll) {
    case 2: return (const void*)seg_strip_kernel<DT, COMP, VB, 2>;
    case 4: return (const void*)seg_strip_kernel<DT, COMP, VB, 4>;
    case 8: return (const void*)seg_strip_kernel<DT, COMP, VB, 8>;
    default: return nullptr;
    }
}

template <int DT, bool COMP, bool DENSE>
inline const void* pick_seg_vec(int vec, int unroll) {
    return vec == 16 ? pick_seg<DT, COMP, 16, DENSE>(unroll)
                     : (vec == 32 ? pick_seg<DT, COMP, 32, DENSE>(unroll) : nullptr);
}

// The three kernel families of one dtype are instantiated in three
// translation units (sr_segmented_<dtype>{,_dense,_bulk}.cu) so they compile
// in parallel.
template <int DT, bool COMP>
inline const void* pick_seg_ldg(int vec, int unroll) { return pick_seg_vec<DT, COMP, false>(vec, unroll); }
template <int DT, bool COMP>
inline const void* pick_seg_dense(int vec, int unroll) { return pick_seg_vec<DT, COMP, true>(vec, unroll); }
template <int DT, bool COMP>
inline const void* pick_seg_tma(int vec, int unroll) {
    return vec == 16 ? pick_seg_bulk<DT, COMP, 16>(unroll) : (vec == 32 ? pick_seg_bulk<DT, COMP, 32>(unroll) : nullptr);
}

// ------------------------------------------------ lane-per-segment form
// Read-only 16-byte load that allocates in L1: for access patterns in which
// neighbouring lanes, or a lane's next load, use the rest of the line.
__device__ __forceinline__ void ldg_vec_l1(const void* p, uint32_t (&r)[4]) {
    asm("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "l"(p));
}
__device__ __forceinline__ void ldg_vec_l1(const void* p, uint32_t (&r)[8]) {
    asm("ld.global.nc.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "l"(p));
}

// One thread sums x[s0, s1) alone: the VB-byte aligned body as VB-byte
// vectors (UNROLL per step, cached in L1: a lane's next vector and its
// neighbours' share the lines), the elements before and after it singly.
template <int DT, bool COMP, int VB, int UNROLL>
__device__ __forceinline__ typename Acc<DT, COMP>::T lane_sum(const unsigned char* x, int64_t s0, int64_t s1) {
    using A = typename Acc<DT, COMP>::T;
    constexpr int EB = SegElem<DT>::v;
    constexpr int PV = VB / EB;  // elements per vector
    constexpr int W = VB / 4;    // 32-bit words per vector
    const uintptr_t xa = reinterpret_cast<uintptr_t>(x);
    int64_t a0 = s0 + (int64_t)((((uintptr_t)VB - (xa + (uintptr_t)s0 * EB) % VB) % VB) / EB);
    if (a0 > s1) a0 = s1;
    const int64_t nv = (s1 - a0) / PV;
    const int64_t a1 = a0 + nv * PV;
    A edge = Op<A>::zero();  // head [s0, a0) and tail [a1, s1), fewer than PV each
    for (int64_t i = s0; i < a0; ++i) acc_elem<DT>(edge, x, i);
    for (int64_t i = a1; i < s1; ++i) acc_elem<DT>(edge, x, i);
    A acc[W];
#pragma unroll
    for (int q = 0; q < W; ++q) acc[q] = Op<A>::zero();
    const unsigned char* body = x + a0 * EB;
    int64_t v = 0;
    for (; v + UNROLL <= nv; v += UNROLL) {
        uint32_t r[UNROLL][W];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) ldg_vec_l1(body + (v + u) * VB, r[u]);
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
#pragma unroll
            for (int q = 0; q < W; ++q) acc_word<DT>(acc[q], r[u][q]);
        }
    }
    for (; v < nv; ++v) {
        uint32_t r[W];
        ldg_vec_l1(body + v * VB, r);
#pragma unroll
        for (int q = 0; q < W; ++q) acc_word<DT>(acc[q], r[q]);
    }
    return Op<A>::add(sum_words<A, W>(acc), edge);
}

// SR_F_LANE_SEGMENTS: thread t of the grid sums segments t, t + T, ... alone
// (T threads), so a warp covers 32 consecutive segments: the offsets and the
// results move as coalesced words, and the lanes' loads fall into the warp's
// contiguous range.  One vector load replaces 16 / element-size scalar
// ones, which cut the time at 16-element segments 2.5-fold.  For very short
// segments only: a thread walks its segment alone.  No grid stage;
// deterministic.
template <int DT, bool COMP, int VB, int UNROLL>
__global__ void __launch_bounds__(512) seg_lane_kernel(const SegParams p) {
    grid_dependency_wait();
    allow_dependents();
    if (p.bad != nullptr && __ldcg(p.bad) != 0) return;  // offsets failed the check: read nothing
    const int64_t T = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < p.nseg; s += T) {
        const int64_t s0 = __ldg(p.offsets + s);
        const int64_t s1 = __ldg(p.offsets + s + 1);
        seg_out(p, s, lane_sum<DT, COMP, VB, UNROLL>(p.x, s0, s1));
    }
}

template <int DT, bool COMP, int VB>
inline const void* pick_seg_lane_u(int unroll) {
    switch (unroll) {
    case 1: return (const void*)seg_lane_kernel<DT, COMP, VB, 1>;
    case 2: return (const void*)seg_lane_kernel<DT, COMP, VB, 2>;
    case 4: return (const void*)seg_lane_kernel<DT, COMP, VB, 4>;
    case 8: return (const void*)seg_lane_kernel<DT, COMP, VB, 8>;
    default: return nullptr;
    }
}
template <int DT, bool COMP>
inline const void* pick_seg_lane(int vec, int unroll) {
    return vec == 16 ? pick_seg_lane_u<DT, COMP, 16>(unroll) : (vec == 32 ? pick_seg_lane_u<DT, COMP, 32>(unroll) : nullptr);
}

// ------------------------------------------------ warp-per-segment form
// SR_F_WARP_SEGMENTS: each warp sums whole segments, so no segment crosses a
// warp and there is no grid stage (results are deterministic).  Warps take
// blocks of G consecutive segments in turn (block b to warp b mod W, G =
// ceil(nseg / W) clamped to 1..32); lane k holds offsets[bG + k], so a block
// costs one coalesced offsets load.  Per segment, the elements before its
// first VB-aligned address and after its last whole vector are single loads
// by the first lanes; the vectors between are spread over the lanes, UNROLL
// per lane and batch; then one warp reduction and one store.  Segments go in
// pairs: both first batches are loaded before either is summed, so each warp
// keeps two segments' loads in flight.  A segment of at most kLaneAloneBytes
// is summed by its own lane instead (lane_sum), all such segments of a block
// at once: skewed layouts, mostly short segments with a long tail, pay the
// warp-wide path only for the long ones.
constexpr int64_t kLaneAloneBytes = 512;  // segments a lane of the warp form sums alone

// One block of nb (<= 32) consecutive segments b0.. summed by one warp: lane
// k holds offsets[b0 + k], so the block costs one coalesced offsets load.
// Segments of at most kLaneAloneBytes are summed by their own lane; the rest
// by the whole warp, two at a time.
template <int DT, bool COMP, int VB, int UNROLL>
__device__ __forceinline__ void seg_warp_block(const SegParams& p, int64_t b0, int64_t nb, int lane) {
    using A = typename Acc<DT, COMP>::T;
    constexpr int EB = SegElem<DT>::v;
    constexpr int PV = VB / EB;  // elements per lane vector
    constexpr int W = VB / 4;    // 32-bit words per lane vector
    const uintptr_t xa = reinterpret_cast<uintptr_t>(p.x);
    const int64_t i = b0 + (lane < nb ? lane : nb);           // lane nb (or 31) holds the end
    const int64_t o = __ldg(p.offsets + i);
    const int64_t o_end = __ldg(p.offsets + b0 + nb);
    // this lane's segment [o, e); the short ones are summed by their lane alone
    const int64_t o_up = __shfl_down_sync(0xffffffffu, o, 1);
    const bool mine = lane < nb;
    const int64_t e = (lane + 1 < nb) ? o_up : o_end;
    const bool alone = mine && (e - o) * EB <= kLaneAloneBytes;
    if (alone) seg_out(p, b0 + lane, lane_sum<DT, COMP, 16, 4>(p.x, o, e));
    // the rest by the whole warp, two at a time: both first batches of loads in flight together
    unsigned todo = __ballot_sync(0xffffffffu, mine && !alone);
    while (todo != 0u) {
        const int k0 = __ffs(todo) - 1;
        todo &= todo - 1u;
        const bool two = todo != 0u;  // warp-uniform
        const int k1 = two ? __ffs(todo) - 1 : k0;
        if (two) todo &= todo - 1u;
        int64_t s0[2], s1[2];
        s0[0] = __shfl_sync(0xffffffffu, o, k0);
        s1[0] = __shfl_sync(0xffffffffu, e, k0);
        s0[1] = __shfl_sync(0xffffffffu, o, k1);
        s1[1] = __shfl_sync(0xffffffffu, e, k1);
        if (!two) s0[1] = s1[1] = s1[0];  // an empty second segment
        int64_t a0[2], nv[2];
        A edge[2], acc[2][W];
        uint32_t r[2][UNROLL][W];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            a0[j] = s0[j] + (int64_t)((((uintptr_t)VB - (xa + (uintptr_t)s0[j] * EB) % VB) % VB) / EB);
            if (a0[j] > s1[j]) a0[j] = s1[j];
            nv[j] = (s1[j] - a0[j]) / PV;
            const int64_t a1 = a0[j] + nv[j] * PV;
            edge[j] = Op<A>::zero();  // head [s0, a0) and tail [a1, s1), fewer than PV each
            if (lane < a0[j] - s0[j]) acc_elem<DT>(edge[j], p.x, s0[j] + lane);
            if (lane < s1[j] - a1) acc_elem<DT>(edge[j], p.x, a1 + lane);
#pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                const int64_t v = u * 32 + lane;
                if (v < nv[j]) ldg_vec(p.x + (a0[j] + v * PV) * EB, r[j][u]);
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
#pragma unroll
            for (int q = 0; q < W; ++q) acc[j][q] = Op<A>::zero();
#pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                if (u * 32 + lane < nv[j]) {
#pragma unroll
                    for (int q = 0; q < W; ++q) acc_word<DT>(acc[j][q], r[j][u][q]);
                }
            }
        }
        // the rest of a segment longer than one batch, with both batch
        // buffers free now: 2 * UNROLL vectors per lane in flight
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const unsigned char* body = p.x + a0[j] * EB;
            for (int64_t v0 = 32 * UNROLL; v0 < nv[j]; v0 += 64 * UNROLL) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int u = 0; u < UNROLL; ++u) {
                        const int64_t v = v0 + (h * UNROLL + u) * 32 + lane;
                        if (v < nv[j]) ldg_vec(body + v * VB, r[h][u]);
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int u = 0; u < UNROLL; ++u) {
                        if (v0 + (h * UNROLL + u) * 32 + lane < nv[j]) {
#pragma unroll
                            for (int q = 0; q < W; ++q) acc_word<DT>(acc[j][q], r[h][u][q]);
                        }
                    }
                }
            }
        }
        const A t0 = warp_reduce(Op<A>::add(sum_words<A, W>(acc[0]), edge[0]));
        const A t1 = warp_reduce(Op<A>::add(sum_words<A, W>(acc[1]), edge[1]));
        if (lane == 0) {
            seg_out(p, b0 + k0, t0);
            if (two) seg_out(p, b0 + k1, t1);
        }
    }
}

template <int DT, bool COMP, int VB, int UNROLL>
__global__ void __launch_bounds__(512) seg_warp_kernel(const SegParams p) {
    grid_dependency_wait();
    allow_dependents();
    if (p.bad != nullptr && __ldcg(p.bad) != 0) return;  // offsets failed the check: read nothing
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t Wn = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int64_t G = (p.nseg + Wn - 1) / Wn;
    G = G < 1 ? 1 : (G > 32 ? 32 : G);
    for (int64_t b0 = w * G; b0 < p.nseg; b0 += Wn * G)
        seg_warp_block<DT, COMP, VB, UNROLL>(p, b0, (p.nseg - b0 < G) ? p.nseg - b0 : G, lane);
}

template <int DT, bool COMP, int VB>
inline const void* pick_seg_warp_u(int unroll) {
    switch (unroll) {
    case 1: return (const void*)seg_warp_kernel<DT, COMP, VB, 1>;
    case 2: return (const void*)seg_warp_kernel<DT, COMP, VB, 2>;
    case 4: return (const void*)seg_warp_kernel<DT, COMP, VB, 4>;
    case 8: return (const void*)seg_warp_kernel<DT, COMP, VB, 8>;
    default: return nullptr;
    }
}
template <int DT, bool COMP>
inline const void* pick_seg_warp(int vec, int unroll) {
    return vec == 16 ? pick_seg_warp_u<DT, COMP, 16>(unroll) : (vec == 32 ? pick_seg_warp_u<DT, COMP, 32>(unroll) : nullptr);
}

}  // namespace sr
