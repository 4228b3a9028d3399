// Small MLP cost model of the learned selector: in_dim -> hidden (ReLU) ->
// hidden (ReLU) -> out_dim logits, softmax cross-entropy against soft target
// distributions, trained with Adam.  All arithmetic runs in these kernels:
//   mlp_grad_kernel   : forward + backward of tiles of eight samples per CTA;
//                       every gradient entry is owned by one thread, and the
//                       CTA's partial gradient is written to its own slot;
//   mlp_update_kernel : sums the CTA partials in a fixed order (deterministic)
//                       and applies one Adam step;
//   mlp_predict_kernel: forward pass and argmax (the inference kernel): one
//                       CTA per sample, weights held in registers, each
//                       layer's dot products split over all 256 threads.
// Parameter layout (row-major, one contiguous float array):
//   W1[in][h], b1[h], W2[h][h], b2[h], W3[h][out], b3[out].
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "sr_device.cuh"
#include "sr_internal.h"

namespace sr {
namespace {

constexpr int kMaxIn = 32, kMaxH = 64, kMaxOut = 64;
constexpr int kThreads = 256;

struct MlpDims {
    int in, h, out;
    int64_t P;
    int64_t oW1, ob1, oW2, ob2, oW3, ob3;
};

MlpDims make_dims(int in, int h, int out) {
    MlpDims d;
    d.in = in;
    d.h = h;
    d.out = out;
    d.oW1 = 0;
    d.ob1 = d.oW1 + (int64_t)in * h;
    d.oW2 = d.ob1 + h;
    d.ob2 = d.oW2 + (int64_t)h * h;
    d.oW3 = d.ob2 + h;
    d.ob3 = d.oW3 + (int64_t)h * out;
    d.P = d.ob3 + out;
    return d;
}

// Gradient kernel.  A batch is a few megaflops, so the step is bound by the
// chain of dependent layers, not by throughput: with one sample at a time it
// was some 10 block barriers and 60-long serial sums per sample, 16 samples in a
// row (146 us a step of the 9-64-40 network at every batch up to 2048; now 9.1 us
// to 256, 10.4 at 1000, 15.9 at 2048, in two launches, bound by shared-memory
// latency).  Here a CTA takes tiles of kTile
// samples through each layer together: thread (column, half of the tile, half of
// the inputs) sums one column for four samples, so a weight is read once for four
// products; the two halves of the inputs meet in shared memory.  The weight
// gradients are outer products summed in registers over all tiles of the CTA
// (thread: 2 rows x 8 columns), the tile's samples in order.  With 128 threads and
// whole columns the same step took 9.8, 11.3 and 16.4 us.
// Layout: weights with a row stride of 65 words (rows and columns are both read
// by 32 lanes without bank conflicts); activations as [feature][kTile], 12 words
// apart (eight consecutive features' float4 fall into different banks).
constexpr int kGradThreads = 256;
constexpr int kTile = 8;    // samples of a tile
constexpr int kWLd = kMaxH + 1;
constexpr int kALd = kTile + 4;

struct GradSmem {  // offsets in floats
    int w1, w2, w3, b1, b2, b3, x, h1, h2, z, dh2, dh1, loss, half, total;
};
__host__ __device__ inline GradSmem grad_smem(const MlpDims& d) {
    GradSmem m;
    int at = 0;
    auto take = [&](int n) {
        const int r = at;
        at += (n + 3) / 4 * 4;
        return r;
    };
    m.w1 = take(d.in * kWLd);
    m.w2 = take(d.h * kWLd);
    m.w3 = take(d.h * kWLd);
    m.b1 = take(kMaxH);
    m.b2 = take(kMaxH);
    m.b3 = take(kMaxOut);
    m.x = take(kMaxIn * kALd);
    m.h1 = take(kMaxH * kALd);
    m.h2 = take(kMaxH * kALd);
    m.z = take(kMaxOut * kALd);  // logits, then their gradient
    m.dh2 = take(kMaxH * kALd);
    m.dh1 = take(kMaxH * kALd);
    m.loss = take(kTile);
    m.half = take(kMaxH * kALd);  // column sums over the second half of the inputs
    m.total = at;
    return m;
}

// One float into shared memory, asynchronously (zero when !valid; src is not read then).
__device__ __forceinline__ void copy_async(float* dst, const float* src, bool valid) {
    const int bytes = valid ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
// Rows [0, rows) of a row-major matrix into shared memory, zero beyond `cols`:
// all copies of the kernel's start are in flight together, one trip to L2.
__device__ __forceinline__ void load_rows(float* dst, const float* __restrict__ src, int rows, int cols) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 4
    for (int r = warp; r < rows; r += kGradThreads / 32) {
#pragma unroll
        for (int c = lane; c < kMaxH; c += 32) copy_async(dst + r * kWLd + c, c < cols ? src + r * cols + c : src, c < cols);
    }
}

// acc[i] += sum_k W(k) * a[k][sg * 4 + i] over k < K; W(k) = w[k * step]
__device__ __forceinline__ void dot4(float (&acc)[4], const float* w, int step, const float* a, int K) {
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
        const float wk = w[k * step];
        const float4 v = *reinterpret_cast<const float4*>(a + k * kALd);
        acc[0] = fmaf(v.x, wk, acc[0]);
        acc[1] = fmaf(v.y, wk, acc[1]);
        acc[2] = fmaf(v.z, wk, acc[2]);
        acc[3] = fmaf(v.w, wk, acc[3]);
    }
}

// g[j][c] += sum over the tile's samples of a[row_j][s] * b[col_c][s], rows
// rg + 32 j, columns cg + 8 c.
template <int NR>
__device__ __forceinline__ void outer(float (&g)[NR][8], const float* a, const float* b, int rg, int cg) {
#pragma unroll 1  // 128 registers: two CTAs per SM
    for (int h = 0; h < kTile; h += 4) {
        float4 u[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) u[j] = *reinterpret_cast<const float4*>(a + (rg + 32 * j) * kALd + h);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float4 v = *reinterpret_cast<const float4*>(b + (cg + 8 * c) * kALd + h);
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                g[j][c] = fmaf(u[j].x, v.x, g[j][c]);
                g[j][c] = fmaf(u[j].y, v.y, g[j][c]);
                g[j][c] = fmaf(u[j].z, v.z, g[j][c]);
                g[j][c] = fmaf(u[j].w, v.w, g[j][c]);
            }
        }
    }
}
template <int NR>
__device__ __forceinline__ void store_grad(float* out, const float (&g)[NR][8], int rows, int cols, int rg, int cg) {
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const int r = rg + 32 * j;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (r < rows && cg + 8 * c < cols) out[r * cols + cg + 8 * c] = g[j][c];
    }
}

__global__ void __launch_bounds__(kGradThreads, 2) mlp_grad_kernel(MlpDims d, const float* __restrict__ params,
                                                                const float* __restrict__ X,
                                                                const float* __restrict__ Q, int B,
                                                                float* __restrict__ partial,
                                                                float* __restrict__ loss_partial) {
    extern __shared__ __align__(16) float sm[];
    const GradSmem m = grad_smem(d);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int col = t & 63, sg = (t >> 6) & 1, kh = t >> 7;  // a column, four samples, half of the inputs
    const int rg = t >> 3, cg = t & 7;                       // weight gradients: rows rg + 32 j, columns cg + 8 c
    grid_dependency_wait();  // the step before may have just written the parameters
    allow_dependents();
    load_rows(sm + m.w1, params + d.oW1, d.in, d.h);
    load_rows(sm + m.w2, params + d.oW2, d.h, d.h);
    load_rows(sm + m.w3, params + d.oW3, d.h, d.out);
    if (t < kMaxH) {
        copy_async(sm + m.b1 + t, params + (t < d.h ? d.ob1 + t : 0), t < d.h);
        copy_async(sm + m.b2 + t, params + (t < d.h ? d.ob2 + t : 0), t < d.h);
        copy_async(sm + m.b3 + t, params + (t < d.out ? d.ob3 + t : 0), t < d.out);
    }
    // rows past the network's own sizes are read by the outer products: zero them once
    for (int i = t; i < m.loss - m.x; i += kGradThreads) sm[m.x + i] = 0.f;
    float g1[1][8] = {}, g2[2][8] = {}, g3[2][8] = {};  // W1 (in <= 32), W2, W3
    float gb[3] = {};                                   // thread t < 64: entry t of b1, b2, b3
    float loss = 0.f;                                   // thread 0
    const float invB = 1.0f / (float)B;
    const int tiles = (B - 1) / kTile + 1;  // B + kTile - 1 may not fit
    __syncthreads();
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int b0 = tile * kTile, nb = min(kTile, B - b0);
        for (int i = t; i < kTile * d.in; i += kGradThreads) {
            const int s = i / d.in, f = i - s * d.in;
            sm[m.x + f * kALd + s] = s < nb ? X[(int64_t)b0 * d.in + i] : 0.f;
        }
        float q[2];  // this warp's sample's targets, for the softmax below
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int o = lane + 32 * h;
            q[h] = (warp < nb && o < d.out) ? Q[(int64_t)(b0 + warp) * d.out + o] : 0.f;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");  // the first tile: the weights
        __syncthreads();
        // a column's sum over K inputs for samples 4 sg .. 4 sg + 3, from `init`: each half
        // of the threads takes half of the inputs, the second leaves its sum in `half`
        float* half = sm + m.half + col * kALd + sg * 4;
        auto half_dot = [&](float (&a)[4], const float* w, int step, const float* src, int K, float init) {
            const int k0 = (K + 1) / 2;
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = kh == 0 ? init : 0.f;
            if (kh == 0) dot4(a, w, step, src + sg * 4, k0);
            else dot4(a, w + k0 * step, step, src + k0 * kALd + sg * 4, K - k0);
            if (kh == 1) *reinterpret_cast<float4*>(half) = make_float4(a[0], a[1], a[2], a[3]);
        };
        auto add_half = [&](float (&a)[4]) {
            const float4 v = *reinterpret_cast<const float4*>(half);
            a[0] += v.x;
            a[1] += v.y;
            a[2] += v.z;
            a[3] += v.w;
        };
        // one layer; samples past the batch are zero
        auto layer = [&](int w, int bias, int src, int K, int dst, bool relu) {
            float a[4];
            half_dot(a, sm + w + col, kWLd, sm + src, K, sm[bias + col]);
            __syncthreads();
            if (kh == 0) {
                add_half(a);
                float4 r;
                float* rv = reinterpret_cast<float*>(&r);
#pragma unroll
                for (int i = 0; i < 4; ++i) rv[i] = (sg * 4 + i < nb && !(relu && !(a[i] > 0.f))) ? a[i] : 0.f;
                *reinterpret_cast<float4*>(sm + dst + col * kALd + sg * 4) = r;
            }
            __syncthreads();
        };
        layer(m.w1, m.b1, m.x, d.in, m.h1, true);
        layer(m.w2, m.b2, m.h1, d.h, m.h2, true);
        layer(m.w3, m.b3, m.h2, d.h, m.z, false);
        // softmax cross-entropy, one sample per warp: z becomes (p - q) / B
        {
            float z[2], mx = -INFINITY;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                z[h] = lane + 32 * h < d.out ? sm[m.z + (lane + 32 * h) * kALd + warp] : -INFINITY;
                mx = fmaxf(mx, z[h]);
            }
            for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            float e = 0.f;
#pragma unroll
            for (int h = 0; h < 2; ++h) e += lane + 32 * h < d.out ? expf(z[h] - mx) : 0.f;
            for (int off = 16; off; off >>= 1) e += __shfl_xor_sync(0xffffffffu, e, off);
            const float lse = mx + logf(e);
            float l = 0.f;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int o = lane + 32 * h;
                if (o < d.out) {
                    sm[m.z + o * kALd + warp] = warp < nb ? (expf(z[h] - lse) - q[h]) * invB : 0.f;
                    l += q[h] * (lse - z[h]);
                }
            }
            for (int off = 16; off; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
            if (lane == 0) sm[m.loss + warp] = warp < nb ? l * invB : 0.f;
        }
        __syncthreads();
        // backward: row `col` of W for the tile's samples, masked by the activation's
        // sign, in two steps around the barrier that the outer product before it shares
        float a[4];
        auto back = [&](int w, int src, int K) {
            if (col < d.h) half_dot(a, sm + w + col * kWLd, 1, sm + src, K, 0.f);
        };
        auto back_end = [&](int act, int dst) {
            __syncthreads();
            if (kh == 0 && col < d.h) {
                add_half(a);
                const float4 h = *reinterpret_cast<const float4*>(sm + act + col * kALd + sg * 4);
                *reinterpret_cast<float4*>(sm + dst + col * kALd + sg * 4) =
                    make_float4(h.x > 0.f ? a[0] : 0.f, h.y > 0.f ? a[1] : 0.f, h.z > 0.f ? a[2] : 0.f,
                                h.w > 0.f ? a[3] : 0.f);
            }
            __syncthreads();
        };
        auto bias_grad = [&](float& g, int src) {
            if (t < kMaxH) {
#pragma unroll
                for (int s = 0; s < kTile; ++s) g += sm[src + t * kALd + s];
            }
        };
        back(m.w3, m.z, d.out);
        outer(g3, sm + m.h2, sm + m.z, rg, cg);
        bias_grad(gb[2], m.z);
        if (t == 0) {
#pragma unroll
            for (int s = 0; s < kTile; ++s) loss += sm[m.loss + s];
        }
        back_end(m.h2, m.dh2);
        back(m.w2, m.dh2, d.h);
        outer(g2, sm + m.h1, sm + m.dh2, rg, cg);
        bias_grad(gb[1], m.dh2);
        back_end(m.h1, m.dh1);
        outer(g1, sm + m.x, sm + m.dh1, rg, cg);
        bias_grad(gb[0], m.dh1);
        __syncthreads();
    }
    float* out = partial + (int64_t)blockIdx.x * d.P;
    store_grad(out + d.oW1, g1, d.in, d.h, rg, cg);
    store_grad(out + d.oW2, g2, d.h, d.h, rg, cg);
    store_grad(out + d.oW3, g3, d.h, d.out, rg, cg);
    if (t < d.h) {
        out[d.ob1 + t] = gb[0];
        out[d.ob2 + t] = gb[1];
    }
    if (t < d.out) out[d.ob3 + t] = gb[2];
    if (t == 0) loss_partial[blockIdx.x] = loss;
}

// Sum the per-CTA partials in a fixed order, optionally export the gradient,
// and (lr > 0) apply Adam: m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2;
// p -= lr * (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps).
// A CTA takes 32 parameters; its warp k sums the partials k, k + 8, ..., warp 0
// adds the eight sums in order (one thread per parameter walked all partials
// alone: with 128 of them, 128 dependent adds behind as many loads).
constexpr int kUpdGroups = 8;

__global__ void __launch_bounds__(32 * kUpdGroups)
    mlp_update_kernel(int64_t P, int nparts, const float* __restrict__ partial, const float* __restrict__ loss_partial,
                      float* params, float* m, float* v, float* __restrict__ grad_out, float* __restrict__ loss_out,
                      float lr, float b1, float b2, float eps, float c1, float c2) {
    __shared__ float part[kUpdGroups][33];
    const int lane = threadIdx.x & 31, group = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    // The state is read before the wait (from L2): the gradient kernel this one
    // follows waited for the update before it, so nothing in flight writes it.
    float mi = 0.f, vi = 0.f, pi = 0.f;
    if (group == 0 && i < P && lr > 0.f) {
        mi = __ldcg(m + i);
        vi = __ldcg(v + i);
        pi = __ldcg(params + i);
    }
    grid_dependency_wait();  // the partials are written
    allow_dependents();
    float s = 0.f;
    if (i < P) {
#pragma unroll 4
        for (int k = group; k < nparts; k += kUpdGroups) s += partial[(int64_t)k * P + i];
    }
    part[group][lane] = s;
    float l = 0.f;
    if (blockIdx.x == 0 && group == 1 && loss_out) {
        for (int k = lane; k < nparts; k += 32) l += loss_partial[k];
        for (int off = 16; off; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        if (lane == 0) *loss_out = l;
    }
    __syncthreads();
    if (group != 0 || i >= P) return;
    float gsum = 0.f;
#pragma unroll
    for (int k = 0; k < kUpdGroups; ++k) gsum += part[k][lane];
    if (grad_out) grad_out[i] = gsum;
    if (lr > 0.f) {
        mi = b1 * mi + (1.f - b1) * gsum;
        vi = b2 * vi + (1.f - b2) * gsum * gsum;
        m[i] = mi;
        v[i] = vi;
        params[i] = pi - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// Inference: one CTA per sample (grid-stride over the batch), 256 threads.
// Each layer's dot products are split four ways: thread (part, col) sums
// rows [part*k, part*k + k) of column col, the four partials meet in shared
// memory and are added in part order (deterministic).  Every thread loads its
// slices of W1, W2 and W3 into registers before anything waits, so the weights
// cost one trip to L2, not one per layer; the 7,400 parameters are never
// staged through shared memory.
constexpr int kParts = 4;
constexpr int kR1 = kMaxIn / kParts, kR2 = kMaxH / kParts;  // rows per part (maximum)

__global__ void __launch_bounds__(kThreads) mlp_predict_kernel(MlpDims d, const float* __restrict__ params,
                                                               const float* __restrict__ X, int B,
                                                               int* __restrict__ cls, float* __restrict__ logits) {
    __shared__ float xs[kMaxIn], h1[kMaxH], h2[kMaxH], z[kMaxOut];
    __shared__ float red[kParts][kMaxH];
    const int tid = threadIdx.x, col = tid & (kMaxH - 1), part = tid / kMaxH;
    const int k1 = (d.in + kParts - 1) / kParts, k2 = (d.h + kParts - 1) / kParts;
    // launched with programmatic stream serialisation: wait for the previous
    // kernel (a training step may have just written the parameters) before
    // any global read; only the launch latency overlaps
    grid_dependency_wait();
    allow_dependents();
    float w1[kR1], w2[kR2], w3[kR2];
#pragma unroll
    for (int r = 0; r < kR1; ++r) {
        const int j = part * k1 + r;
        w1[r] = (r < k1 && j < d.in && col < d.h) ? __ldg(params + d.oW1 + (int64_t)j * d.h + col) : 0.f;
    }
#pragma unroll
    for (int r = 0; r < kR2; ++r) {
        const int j = part * k2 + r;
        const bool row = r < k2 && j < d.h;
        w2[r] = (row && col < d.h) ? __ldg(params + d.oW2 + (int64_t)j * d.h + col) : 0.f;
        w3[r] = (row && col < d.out) ? __ldg(params + d.oW3 + (int64_t)j * d.out + col) : 0.f;
    }
    const float bias1 = (part == 0 && col < d.h) ? __ldg(params + d.ob1 + col) : 0.f;
    const float bias2 = (part == 0 && col < d.h) ? __ldg(params + d.ob2 + col) : 0.f;
    const float bias3 = (part == 0 && col < d.out) ? __ldg(params + d.ob3 + col) : 0.f;

    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        if (tid < d.in) xs[tid] = X[(int64_t)b * d.in + tid];
        __syncthreads();
        float a = 0.f;
#pragma unroll
        for (int r = 0; r < kR1; ++r)
            if (r < k1 && part * k1 + r < d.in) a = fmaf(xs[part * k1 + r], w1[r], a);
        red[part][col] = a;
        __syncthreads();
        if (tid < d.h) {
            const float v = ((bias1 + red[0][tid]) + red[1][tid]) + (red[2][tid] + red[3][tid]);
            h1[tid] = v > 0.f ? v : 0.f;
        }
        __syncthreads();
        a = 0.f;
#pragma unroll
        for (int r = 0; r < kR2; ++r)
            if (r < k2 && part * k2 + r < d.h) a = fmaf(h1[part * k2 + r], w2[r], a);
        red[part][col] = a;
        __syncthreads();
        if (tid < d.h) {
            const float v = ((bias2 + red[0][tid]) + red[1][tid]) + (red[2][tid] + red[3][tid]);
            h2[tid] = v > 0.f ? v : 0.f;
        }
        __syncthreads();
        a = 0.f;
#pragma unroll
        for (int r = 0; r < kR2; ++r)
            if (r < k2 && part * k2 + r < d.h) a = fmaf(h2[part * k2 + r], w3[r], a);
        red[part][col] = a;
        __syncthreads();
        if (tid < d.out) {
            z[tid] = ((bias3 + red[0][tid]) + red[1][tid]) + (red[2][tid] + red[3][tid]);
            if (logits) logits[(int64_t)b * d.out + tid] = z[tid];
        }
        __syncthreads();
        if (tid < 32) {  // argmax, lowest index on ties
            float best = -INFINITY;
            int bi = d.out;
            for (int o = tid; o < d.out; o += 32)
                if (z[o] > best) {
                    best = z[o];
                    bi = o;
                }
            for (int off = 16; off; off >>= 1) {
                const float ob = __shfl_xor_sync(0xffffffffu, best, off);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
                if (ob > best || (ob == best && oi < bi)) {
                    best = ob;
                    bi = oi;
                }
            }
            if (tid == 0) cls[b] = bi;
        }
        // the next sample's xs write is behind the barrier after it; z and
        // red are rewritten only behind later barriers
    }
}

}  // namespace
}  // namespace sr

using namespace sr;

struct sr_mlp_s {
    MlpDims d;
    float* params = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    float* partial = nullptr;
    float* loss_partial = nullptr;
    int max_parts = 0;
    int step = 0;
};

extern "C" {

int sr_mlp_create(int in_dim, int hidden, int out_dim, sr_mlp* out) {
    if (!out || in_dim < 1 || in_dim > kMaxIn || hidden < 1 || hidden > kMaxH || out_dim < 2 || out_dim > kMaxOut)
        return SR_ERR_ARG;
    *out = nullptr;
    sr_mlp h = new sr_mlp_s;
    h->d = make_dims(in_dim, hidden, out_dim);
    const size_t pb = sizeof(float) * (size_t)h->d.P;
    cudaError_t e = cudaMalloc(&h->params, pb);
    if (e == cudaSuccess) e = cudaMalloc(&h->m, pb);
    if (e == cudaSuccess) e = cudaMalloc(&h->v, pb);
    if (e == cudaSuccess) e = cudaMemset(h->params, 0, pb);
    if (e == cudaSuccess) e = cudaMemset(h->m, 0, pb);
    if (e == cudaSuccess) e = cudaMemset(h->v, 0, pb);
    if (e != cudaSuccess) {
        sr_mlp_destroy(h);
        return status_from_cuda(e);
    }
    *out = h;
    return SR_OK;
}

int sr_mlp_destroy(sr_mlp h) {
    if (!h) return SR_OK;
    cudaFree(h->params);
    cudaFree(h->m);
    cudaFree(h->v);
    cudaFree(h->partial);
    cudaFree(h->loss_partial);
    delete h;
    return SR_OK;
}

int64_t sr_mlp_param_count(sr_mlp h) { return h ? h->d.P : -SR_ERR_ARG; }

int sr_mlp_dims(sr_mlp h, int* in_dim, int* hidden, int* out_dim) {
    if (!h || !in_dim || !hidden || !out_dim) return SR_ERR_ARG;
    *in_dim = h->d.in;
    *hidden = h->d.h;
    *out_dim = h->d.out;
    return SR_OK;
}

int sr_mlp_set_params(sr_mlp h, const float* host, int64_t count) {
    if (!h || !host || count != h->d.P) return SR_ERR_ARG;
    cudaError_t e = cudaMemcpy(h->params, host, sizeof(float) * count, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(h->m, 0, sizeof(float) * count);
    if (e == cudaSuccess) e = cudaMemset(h->v, 0, sizeof(float) * count);
    h->step = 0;
    return e == cudaSuccess ? SR_OK : status_from_cuda(e);
}

int sr_mlp_get_params(sr_mlp h, float* host, int64_t count) {
    if (!h || !host || count != h->d.P) return SR_ERR_ARG;
    cudaError_t e = cudaMemcpy(host, h->params, sizeof(float) * count, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? SR_OK : status_from_cuda(e);
}

int sr_mlp_train_step(sr_mlp h, const float* X, const float* Q, int batch, float lr, float* loss, float* grad,
                      sr_stream_t stream) {
    if (!h || !X || !Q || batch < 1 || !(lr >= 0.f)) return SR_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    int st = SR_OK;
    const DeviceInfo* di = current_device(&st);
    if (!di) return st;
    // one tile of samples per CTA up to two CTAs per SM, then several
    const int parts = (int)std::min<int64_t>(((int64_t)batch + kTile - 1) / kTile, 2 * di->sms);
    cudaError_t e;
    if (parts > h->max_parts) {
        // room for every batch up to the next multiple of 16, so that a step captured
        // after one of a slightly smaller batch need not allocate
        const int room = (int)std::min<int64_t>(2 * (((int64_t)batch + 15) / 16), 2 * di->sms);
        cudaFree(h->partial);
        cudaFree(h->loss_partial);
        h->partial = nullptr;
        h->loss_partial = nullptr;
        e = cudaMalloc(&h->partial, sizeof(float) * (size_t)room * h->d.P);
        if (e == cudaSuccess) e = cudaMalloc(&h->loss_partial, sizeof(float) * room);
        if (e != cudaSuccess) {
            h->max_parts = 0;
            return status_from_cuda(e);
        }
        h->max_parts = room;
    }
    const size_t smem = sizeof(float) * (size_t)grad_smem(h->d).total;
    st = prepare_function((const void*)mlp_grad_kernel, smem, false);
    if (st != SR_OK) return st;
    // programmatic stream serialisation: each kernel is scheduled while the one
    // before it drains and waits for it before its first global read
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc;
    std::memset(&lc, 0, sizeof lc);
    lc.gridDim = dim3((unsigned)parts);
    lc.blockDim = dim3(kGradThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    lc.attrs = pdl;
    lc.numAttrs = 1;
    e = cudaLaunchKernelEx(&lc, mlp_grad_kernel, h->d, (const float*)h->params, X, Q, batch, h->partial,
                           h->loss_partial);
    if (e != cudaSuccess) return status_from_cuda(e);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    if (lr > 0.f) h->step += 1;
    const float c1 = lr > 0.f ? 1.f - powf(b1, (float)h->step) : 1.f;
    const float c2 = lr > 0.f ? 1.f - powf(b2, (float)h->step) : 1.f;
    lc.gridDim = dim3((unsigned)((h->d.P + 31) / 32));
    lc.blockDim = dim3(32 * kUpdGroups);
    lc.dynamicSmemBytes = 0;
    e = cudaLaunchKernelEx(&lc, mlp_update_kernel, h->d.P, parts, (const float*)h->partial,
                           (const float*)h->loss_partial, h->params, h->m, h->v, grad, loss, lr, b1, b2, eps, c1, c2);
    return e == cudaSuccess ? SR_OK : status_from_cuda(e);
}

int sr_mlp_predict(sr_mlp h, const float* X, int batch, int* cls, float* logits, sr_stream_t stream) {
    if (!h || !X || !cls || batch < 1) return SR_ERR_ARG;
    const int blocks = batch < 4096 ? batch : 4096;  // one CTA per sample, grid-stride beyond
    cudaLaunchConfig_t lc;
    std::memset(&lc, 0, sizeof lc);
    lc.gridDim = dim3(blocks);
    lc.blockDim = dim3(kThreads);
    lc.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    const MlpDims dd = h->d;
    const float* prm = h->params;
    void* args[] = {const_cast<MlpDims*>(&dd), const_cast<float**>(&prm), const_cast<float**>(&X), &batch, &cls,
                    &logits};
    cudaError_t le = cudaLaunchKernelExC(&lc, (const void*)mlp_predict_kernel, args);
    if (le != cudaSuccess) return status_from_cuda(le);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SR_OK : status_from_cuda(e);
}

}  // extern "C"
