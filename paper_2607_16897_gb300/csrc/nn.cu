// Learned initial-pose proposal: a 3 x (conv 3x3 stride 2 pad 1 + ReLU) +
// 2-layer MLP network (189064 parameters) mapping the coarsest-level residual
// image (1 x 30 x 40) and the previous inter-frame motion (6) to an 8-vector
// increment of the initial state.  Hand-written training and inference
// kernels: BF16 weights (rounded from FP32 master weights after every Adam
// step), FP32 activations and accumulation, deterministic reductions (fixed
// summation order, no atomics).
//
// Flat parameter layout: conv1.w [16,1,3,3], conv1.b [16], conv2.w [32,16,3,3],
// conv2.b [32], conv3.w [64,32,3,3], conv3.b [64], fc1.w [128,1286],
// fc1.b [128], fc2.w [8,128], fc2.b [8], row-major, in that order.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>

#include "glt_internal.h"

namespace glt {
namespace nn {

constexpr int kIn = 1200, kMotion = 6, kOut = 8, kFlat = 1280, kF = 1286, kHid = 128;
struct Layer {
    int w, b;  // offsets of weight and bias in the flat layout
};
constexpr Layer kC1 = {0, 144}, kC2 = {160, 4768}, kC3 = {4800, 23232}, kF1 = {23296, 187904},
                kF2 = {188032, 189056};
constexpr int kParams = 189064;

__device__ __forceinline__ float wv(const __nv_bfloat16* w, int i) { return __bfloat162float(w[i]); }

// BF16 weights in the layouts the kernels read, rewritten with every change of
// the BF16 copy: conv2 and conv3 as [input channel x tap][output channel] (the
// forward pass), the same two as [output channel][tap][input channel] (the
// input gradients), fc1 as [input][output].
constexpr int kW2 = 144 * 32, kW3 = 288 * 64, kW4 = kF * kHid;
constexpr int kT2 = 0, kT3 = kT2 + kW2, kB2 = kT3 + kW3, kB3 = kB2 + kW2, kT4 = kB3 + kW3, kWt = kT4 + kW4;
static_assert(kT3 % 8 == 0 && kB2 % 8 == 0 && kB3 % 8 == 0 && kT4 % 8 == 0, "16-byte aligned parts");

// Parameter i's places in the relayouted copy.
__device__ __forceinline__ void put_wt(__nv_bfloat16* __restrict__ wt, int i, __nv_bfloat16 v)
{
    if (i >= kC2.w && i < kC2.w + kW2) {
        const int q = i - kC2.w, o = q / 144, k = q % 144;       // k = c * 9 + tap
        wt[kT2 + k * 32 + o] = v;
        wt[kB2 + (o * 9 + k % 9) * 16 + k / 9] = v;
    } else if (i >= kC3.w && i < kC3.w + kW3) {
        const int q = i - kC3.w, o = q / 288, k = q % 288;
        wt[kT3 + k * 64 + o] = v;
        wt[kB3 + (o * 9 + k % 9) * 32 + k / 9] = v;
    } else if (i >= kF1.w && i < kF1.w + kW4) {
        const int q = i - kF1.w;
        wt[kT4 + (q % kF) * kHid + q / kF] = v;
    }
}

// Bordered activation planes keep each row as its even columns followed by
// its odd columns (column c of a row of Wp at (c & 1) * Wp / 2 + c / 2): the
// stride-2 3x3 windows of consecutive output pixels then read consecutive
// words, where the plain layout reads every other one (two-way bank
// conflicts).
__device__ __forceinline__ int split_col(int c, int Wp) { return (c & 1) * (Wp >> 1) + (c >> 1); }

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem)
{
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

// Two FP32 FMAs in one instruction (fma.rn.f32x2, each half rounded as fmaf
// does): the pipe's rate is the same, but one issue slot serves both.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ float2 bf2(unsigned v) { return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v)); }

__device__ __forceinline__ f32x2 bfx2(unsigned v)
{
    return pack2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}

// ---------------------------------------------------------------------------
// Forward pass, convolutions: one persistent block per SM runs conv1-conv3 of
// S samples at a time with all activations and the BF16 weights in shared
// memory, so a sample costs its 4.8 KB of input and 5 KB of features in HBM.
// Bound by FP32 issue: conv2 and conv3 are 5-pixel x CH-channel register tiles
// (a window row's 11 values loaded once for its 15 uses, 3 weight loads; the
// lanes of a warp share their weights), conv3 in two halves of its input
// channels, conv1 8 channels of one pixel.  S = 4 fills the
// shared memory and has the larger tiles; S = 2 has twice the blocks, and is
// taken while those still fit one round (kFwdSmall; 256 samples 31 us, 39 with S =
// 4; 305 samples 50, 43 with S = 4).  Training also
// stores the activations (a1, a2) that the backward pass reads.  5000 samples:
// 2.03 ms by one thread per output on global memory, 0.27 ms here; 256: 139 ->
// 24 us (caches flushed).
// ---------------------------------------------------------------------------
constexpr int kFwdThreads = 512;
constexpr int kXs = 32 * 42 + 16, kA1s = 16 * 17 * 22 + 2, kA2s = 32 * 10 * 12 + 1;   // per sample (banks: conv_tiles)
constexpr int kFwdSmall = 2;        // samples per block of the small form

template <int S>
struct FwdSmem {
    float x[S * kXs], a1[S * kA1s], a2[S * kA2s];
    alignas(16) float w1[9 * 16];
    float b1[16], b2[32], b3[64];
    alignas(16) __nv_bfloat16 w2[kW2], w3[kW3];
};
static_assert(5 * 256 <= kXs, "conv3's partial sums (5 S x 256 floats) go over x, which is no longer needed");
static_assert(offsetof(FwdSmem<2>, w3) == offsetof(FwdSmem<2>, w2) + kW2 * sizeof(__nv_bfloat16) &&
                  offsetof(FwdSmem<4>, w3) == offsetof(FwdSmem<4>, w2) + kW2 * sizeof(__nv_bfloat16) &&
                  offsetof(FwdSmem<2>, w3) % 16 == 0 && offsetof(FwdSmem<4>, w3) % 16 == 0 &&
                  offsetof(FwdSmem<4>, a2) == (size_t)4 * (kXs + kA1s) * sizeof(float),
              "one 16-byte aligned weight copy; contiguous planes");

// stride-2 3x3 conv + bias + ReLU of S samples from bordered, column-split
// planes: a thread computes 5 neighbouring pixels of a row x CH channels of one
// sample.  Their 15 window values of a row are 11 different ones, loaded once;
// the lanes of a warp take the rows (two halves of a row for the 10-pixel
// ones) of two or more samples, and the sample strides place their words in
// different banks (rows 24 or 44 words apart, halves 5, samples 1 or 2).
// KS: the input channels in KS parts, one per thread group; part 0 adds the
// others' sums through `red` (shared memory).
template <int S, int C, int W, int HO, int WO, int O, int CH, int IN, int KS, class Out>
__device__ __forceinline__ void conv_tiles(const float* __restrict__ in, const __nv_bfloat16* __restrict__ w,
                                           const float* __restrict__ bias, float* __restrict__ red, Out out)
{
    constexpr int Wp = W + 2, plane = (2 * HO + (W == 20 ? 1 : 2)) * Wp, half = Wp / 2;
    constexpr int PT = 5, PR = WO / PT, PG = HO * PR;
    constexpr int NT = S * PG * (O / CH);
    static_assert(NT * KS == kFwdThreads, "one tile per thread");
    const int t = threadIdx.x % NT, ks = threadIdx.x / NT;
    const int pg = t % PG, s = (t / PG) % S, cg = t / (PG * S);
    const int i = pg / PR, j = (pg % PR) * PT;
    const float* xb = in + s * IN + 2 * i * Wp + j;          // window row 2i, split column of 2j
    f32x2 acc[PT][CH / 2];
#pragma unroll
    for (int k = 0; k < CH / 2; ++k) {
        const f32x2 b = ks ? 0ull : pack2(bias[cg * CH + 2 * k], bias[cg * CH + 2 * k + 1]);
#pragma unroll
        for (int u = 0; u < PT; ++u) acc[u][k] = b;
    }
#pragma unroll 1
    for (int c = ks * (C / KS); c < (ks + 1) * (C / KS); ++c) {
#pragma unroll
        for (int di = 0; di < 3; ++di) {
            const float* xr = xb + c * plane + di * Wp;
            f32x2 ev[PT + 1], od[PT];
#pragma unroll
            for (int u = 0; u <= PT; ++u) ev[u] = pack2(xr[u], xr[u]);                 // columns 2j, 2j + 2, ..
#pragma unroll
            for (int u = 0; u < PT; ++u) od[u] = pack2(xr[half + u], xr[half + u]);    // columns 2j + 1, ..
#pragma unroll
            for (int dj = 0; dj < 3; ++dj) {
                const __nv_bfloat16* wq = w + (c * 9 + di * 3 + dj) * O + cg * CH;
                f32x2 wf[CH / 2];
                if constexpr (CH == 8) {
                    const uint4 r = *reinterpret_cast<const uint4*>(wq);
                    wf[0] = bfx2(r.x), wf[1] = bfx2(r.y), wf[2] = bfx2(r.z), wf[3] = bfx2(r.w);
                } else if constexpr (CH == 4) {
                    const uint2 r = *reinterpret_cast<const uint2*>(wq);
                    wf[0] = bfx2(r.x), wf[1] = bfx2(r.y);
                } else {
                    wf[0] = bfx2(*reinterpret_cast<const unsigned*>(wq));
                }
#pragma unroll
                for (int u = 0; u < PT; ++u) {
                    const f32x2 a = dj == 0 ? ev[u] : dj == 1 ? od[u] : ev[u + 1];
#pragma unroll
                    for (int k = 0; k < CH / 2; ++k) acc[u][k] = fma2(wf[k], a, acc[u][k]);
                }
            }
        }
    }
    if constexpr (KS == 2) {
        if (ks) {
#pragma unroll
            for (int u = 0; u < PT; ++u)
#pragma unroll
                for (int k = 0; k < CH / 2; ++k) {
                    const float2 r = unpack2(acc[u][k]);
                    red[(u * CH + 2 * k) * NT + t] = r.x;
                    red[(u * CH + 2 * k + 1) * NT + t] = r.y;
                }
        }
        __syncthreads();
        if (ks) return;
    }
#pragma unroll
    for (int u = 0; u < PT; ++u)
#pragma unroll
        for (int k = 0; k < CH / 2; ++k) {
            float2 r = unpack2(acc[u][k]);
            if constexpr (KS == 2) {
                r.x += red[(u * CH + 2 * k) * NT + t];
                r.y += red[(u * CH + 2 * k + 1) * NT + t];
            }
            out(s, cg * CH + 2 * k, i * WO + j + u, fmaxf(r.x, 0.0f));
            out(s, cg * CH + 2 * k + 1, i * WO + j + u, fmaxf(r.y, 0.0f));
        }
}

template <int S, bool TRAIN>
__global__ void __launch_bounds__(kFwdThreads, 1)
conv_forward(const float* __restrict__ x, const __nv_bfloat16* __restrict__ w, const __nv_bfloat16* __restrict__ wt,
             int B, float* __restrict__ a1g, float* __restrict__ a2g, float* __restrict__ a3g)
{
    extern __shared__ __align__(16) unsigned char raw[];
    FwdSmem<S>& M = *reinterpret_cast<FwdSmem<S>*>(raw);
    const int tid = threadIdx.x;
    for (int v = tid; v < (kW2 + kW3) / 8; v += kFwdThreads) cp_async16(M.w2 + 8 * v, wt + kT2 + 8 * v);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    for (int i = tid; i < 144; i += kFwdThreads) M.w1[(i % 9) * 16 + i / 9] = wv(w, kC1.w + i);
    if (tid < 16) M.b1[tid] = wv(w, kC1.b + tid);
    if (tid < 32) M.b2[tid] = wv(w, kC2.b + tid);
    if (tid < 64) M.b3[tid] = wv(w, kC3.b + tid);
    // zero borders: cleared once, the interiors are rewritten for every group
    for (int i = tid; i < S * (kXs + kA1s + kA2s); i += kFwdThreads) M.x[i] = 0.0f;
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    // a group's inputs, loaded while the group before it is computed
    constexpr int NX = (S * kIn + kFwdThreads - 1) / kFwdThreads;
    float xv[NX];
    auto load = [&](int b0) {
#pragma unroll
        for (int q = 0; q < NX; ++q) {
            const int i = tid + q * kFwdThreads;
            xv[q] = i < S * kIn && (size_t)b0 * kIn + i < (size_t)B * kIn ? x[(size_t)b0 * kIn + i] : 0.0f;
        }
    };
    load(blockIdx.x * S);
    for (int b0 = blockIdx.x * S; b0 < B; b0 += gridDim.x * S) {
        // (conv3's partial sums went over the planes' borders)
        for (int i = tid; i < S * 144; i += kFwdThreads) {
            const int s = i / 144, e = i % 144;
            const int r = e < 84 ? (e / 42) * 31 : 1 + (e - 84) / 2, c = e < 84 ? e % 42 : ((e - 84) & 1) * 41;
            M.x[s * kXs + r * 42 + split_col(c, 42)] = 0.0f;
        }
#pragma unroll
        for (int q = 0; q < NX; ++q) {
            const int i = tid + q * kFwdThreads, s = i / kIn, p = i - s * kIn, r = p / 40, c = p - r * 40;
            if (i < S * kIn) M.x[s * kXs + (r + 1) * 42 + split_col(c + 1, 42)] = xv[q];
        }
        __syncthreads();
        if (b0 + (int)gridDim.x * S < B) load(b0 + gridDim.x * S);
        for (int t = tid; t < S * 600; t += kFwdThreads) {
            const int p = t % 300, s = (t / 300) % S, og = t / (300 * S), i = p / 20, j = p % 20;
            const float* xb = M.x + s * kXs + 2 * i * 42 + j;
            float acc[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = M.b1[og * 8 + k];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const float v = xb[(q / 3) * 42 + ((q % 3) & 1) * 21 + ((q % 3) >> 1)];
                const float4 wa = *reinterpret_cast<const float4*>(&M.w1[q * 16 + og * 8]);
                const float4 wb = *reinterpret_cast<const float4*>(&M.w1[q * 16 + og * 8 + 4]);
                const float wk[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
                for (int k = 0; k < 8; ++k) acc[k] = fmaf(wk[k], v, acc[k]);
            }
            const int at = s * kA1s + (i + 1) * 22 + split_col(j + 1, 22);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int o = og * 8 + k;
                const float r = fmaxf(acc[k], 0.0f);
                M.a1[at + o * 374] = r;
                if (TRAIN && b0 + s < B) a1g[((size_t)(b0 + s) * 16 + o) * 300 + p] = r;
            }
        }
        __syncthreads();
        conv_tiles<S, 16, 20, 8, 10, 32, S, kA1s, 1>(M.a1, M.w2, M.b2, nullptr, [&](int s, int o, int p, float r) {
            M.a2[s * kA2s + o * 120 + (p / 10 + 1) * 12 + split_col(p % 10 + 1, 12)] = r;
            if (TRAIN && b0 + s < B) a2g[((size_t)(b0 + s) * 32 + o) * 80 + p] = r;
        });
        __syncthreads();
        conv_tiles<S, 32, 10, 4, 5, 64, S, kA2s, 2>(M.a2, M.w3, M.b3, M.x, [&](int s, int o, int p, float r) {
            if (b0 + s < B) a3g[(size_t)(b0 + s) * kFlat + o * 20 + p] = r;
        });
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Fully connected layers.  fc1 tiles 4 samples x 4 outputs (or 8 x 4) per
// thread over the transposed BF16 weights and the features in shared memory;
// then fc2 and, in training, the loss terms, dy = (y - t) / B and fc2's input
// gradient dh (with fc1's ReLU mask).  Two forms:
//  * fc_forward_split, for few samples (a chip's worth of blocks matters more
//    than reuse): a cluster of 8 blocks shares 8 samples, each block summing an
//    eighth of the 1286 inputs; the partial sums meet through distributed
//    shared memory in rank order and each block finishes one sample;
//  * fc_forward_tile, for many: 32 samples per block, the inputs staged 64 at
//    a time with two stages of asynchronous copies.
// ---------------------------------------------------------------------------
constexpr int kFcS = 8;

// fc2 of one sample from its hidden vector hs: 8 warps, one output each
template <bool TRAIN>
__device__ __forceinline__ void fc2_sample(const float* __restrict__ hs, float* __restrict__ ys, const __nv_bfloat16* __restrict__ w,
                                           int b, int B, float* __restrict__ y, const float* __restrict__ t)
{
    const int lane = threadIdx.x & 31, o = threadIdx.x >> 5;
    float v = 0.0f;
#pragma unroll
    for (int i = 0; i < kHid / 32; ++i) v = fmaf(wv(w, kF2.w + o * kHid + lane + 32 * i), hs[lane + 32 * i], v);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    v += wv(w, kF2.b + o);
    if (lane == 0) {
        if (!TRAIN)
            y[(size_t)b * kOut + o] = v;
        else
            ys[o] = v - t[(size_t)b * kOut + o];
    }
}

// loss term, dy and dh of one sample from its errors ys (256 threads; after a barrier)
__device__ __forceinline__ void fc2_backward(const float* __restrict__ hs, const float* __restrict__ ys,
                                             const __nv_bfloat16* __restrict__ w, int b, int B, float* __restrict__ h,
                                             float* __restrict__ dy, float* __restrict__ dh, float* __restrict__ loss_b)
{
    const int tid = threadIdx.x;
    if (tid < kHid) {
        float v = 0.0f;
#pragma unroll
        for (int o = 0; o < kOut; ++o) v = fmaf(wv(w, kF2.w + o * kHid + tid), ys[o] / (float)B, v);
        h[(size_t)b * kHid + tid] = hs[tid];
        dh[(size_t)b * kHid + tid] = hs[tid] > 0.0f ? v : 0.0f;
    } else if (tid < kHid + kOut) {
        dy[(size_t)b * kOut + tid - kHid] = ys[tid - kHid] / (float)B;
    } else if (tid == kHid + kOut) {
        float e = 0.0f;
#pragma unroll
        for (int o = 0; o < kOut; ++o) e = fmaf(ys[o], ys[o], e);
        loss_b[b] = e;
    }
}

constexpr int kSpC = 8, kSpK = 162, kSpThreads = 256;       // cluster, inputs per block
static_assert(kSpC * kSpK >= kF && kSpC == kFcS && kSpThreads / 32 == kOut, "one sample per block, one output per warp");

struct SplitSmem {
    __nv_bfloat16 w[kSpK * kHid];
    float f[kSpK * kFcS];                        // [input][sample]
    float part[kSpThreads / 32][kFcS][kHid];     // the warps' sums
    float sum[kFcS][kHid];                       // the block's
    float hs[kHid], ys[kOut];
};

static_assert(offsetof(SplitSmem, f) % 16 == 0 && offsetof(SplitSmem, part) % 16 == 0, "16-byte accesses");

template <bool TRAIN>
__global__ void __launch_bounds__(kSpThreads)
fc_forward_split(const float* __restrict__ a3, const float* __restrict__ mo, const __nv_bfloat16* __restrict__ w,
                 const __nv_bfloat16* __restrict__ wt, int B, float* __restrict__ y, const float* __restrict__ t,
                 float* __restrict__ h, float* __restrict__ dy, float* __restrict__ dh, float* __restrict__ loss_b)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char raw[];
    SplitSmem& M = *reinterpret_cast<SplitSmem*>(raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cluster.block_rank(), b0 = (blockIdx.x / kSpC) * kFcS;
    const int k0 = rank * kSpK, nk = min(kSpK, kF - k0);
    for (int i = tid; i < nk * (kHid / 8); i += kSpThreads) cp_async16(M.w + 8 * i, wt + kT4 + k0 * kHid + 8 * i);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
#pragma unroll
    for (int q = 0; q < (kFcS * kSpK + kSpThreads - 1) / kSpThreads; ++q) {
        const int i = tid + q * kSpThreads, s = i / kSpK, kk = i - s * kSpK, k = k0 + kk;
        if (i < kFcS * kSpK) {
            float v = 0.0f;
            if (b0 + s < B && k < kF)
                v = k < kFlat ? a3[(size_t)(b0 + s) * kFlat + k] : mo[(size_t)(b0 + s) * kMotion + (k - kFlat)];
            M.f[kk * kFcS + s] = v;
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    // 4 outputs x 8 samples per thread, the warps on consecutive eighths of the block's inputs
    f32x2 acc[kFcS][2];
#pragma unroll
    for (int s = 0; s < kFcS; ++s) acc[s][0] = acc[s][1] = 0ull;
    constexpr int KW = (kSpK + 7) / 8;
    const int ke = min(nk, (warp + 1) * KW);
#pragma unroll 3
    for (int k = warp * KW; k < ke; ++k) {
        const uint2 r = *reinterpret_cast<const uint2*>(M.w + k * kHid + 4 * lane);
        const f32x2 wa = bfx2(r.x), wb = bfx2(r.y);
        const float4 fa = *reinterpret_cast<const float4*>(M.f + k * kFcS);
        const float4 fb = *reinterpret_cast<const float4*>(M.f + k * kFcS + 4);
        const float fs[kFcS] = {fa.x, fa.y, fa.z, fa.w, fb.x, fb.y, fb.z, fb.w};
#pragma unroll
        for (int s = 0; s < kFcS; ++s) {
            const f32x2 v = pack2(fs[s], fs[s]);
            acc[s][0] = fma2(wa, v, acc[s][0]);
            acc[s][1] = fma2(wb, v, acc[s][1]);
        }
    }
#pragma unroll
    for (int s = 0; s < kFcS; ++s) {
        const float2 a = unpack2(acc[s][0]), b = unpack2(acc[s][1]);
        *reinterpret_cast<float4*>(&M.part[warp][s][4 * lane]) = make_float4(a.x, a.y, b.x, b.y);
    }
    __syncthreads();
    for (int i = tid; i < kFcS * kHid; i += kSpThreads) {
        float v = 0.0f;
#pragma unroll
        for (int q = 0; q < kSpThreads / 32; ++q) v += (&M.part[q][0][0])[i];
        (&M.sum[0][0])[i] = v;
    }
    cluster.sync();
    const int b = b0 + rank;                     // this block's sample
    if (tid < kHid) {
        float p[kSpC], v = 0.0f;
#pragma unroll
        for (int q = 0; q < kSpC; ++q) p[q] = cluster.map_shared_rank(&M.sum[rank][0], q)[tid];
#pragma unroll
        for (int q = 0; q < kSpC; ++q) v += p[q];
        M.hs[tid] = fmaxf(v + wv(w, kF1.b + tid), 0.0f);
    }
    // every partial has been read: a block may leave
    cluster.sync();
    if (b >= B) return;
    fc2_sample<TRAIN>(M.hs, M.ys, w, b, B, y, t);
    if (!TRAIN) return;
    __syncthreads();
    fc2_backward(M.hs, M.ys, w, b, B, h, dy, dh, loss_b);
}

constexpr int kTlS = 32, kTlK = 64, kTlThreads = 256;

struct TileSmem {
    __nv_bfloat16 w[2][kTlK * kHid];
    float f[2][kTlS * kTlK];                     // [sample][input]
    float hs[kTlS][kHid], ys[kTlS][kOut];
};

static_assert(offsetof(TileSmem, f) % 16 == 0, "16-byte accesses");

template <bool TRAIN>
__global__ void __launch_bounds__(kTlThreads)
fc_forward_tile(const float* __restrict__ a3, const float* __restrict__ mo, const __nv_bfloat16* __restrict__ w,
                const __nv_bfloat16* __restrict__ wt, int B, float* __restrict__ y, const float* __restrict__ t,
                float* __restrict__ h, float* __restrict__ dy, float* __restrict__ dh, float* __restrict__ loss_b)
{
    extern __shared__ __align__(16) unsigned char raw[];
    TileSmem& M = *reinterpret_cast<TileSmem*>(raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b0 = blockIdx.x * kTlS, nb = min(kTlS, B - b0);
    auto stage = [&](int st, int k0) {
#pragma unroll
        for (int q = 0; q < kTlK * kHid / 8 / kTlThreads; ++q) {
            const int i = tid + q * kTlThreads;
            cp_async16(M.w[st] + 8 * i, wt + kT4 + k0 * kHid + 8 * i);
        }
#pragma unroll
        for (int q = 0; q < kTlS * kTlK / 4 / kTlThreads; ++q) {
            const int i = tid + q * kTlThreads, s = i / (kTlK / 4), c = i % (kTlK / 4);
            cp_async16(M.f[st] + s * kTlK + 4 * c, a3 + (size_t)(b0 + min(s, nb - 1)) * kFlat + k0 + 4 * c);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    // samples 4 warp .. + 3, outputs 4 lane .. + 3
    f32x2 acc[4][2];
#pragma unroll
    for (int s = 0; s < 4; ++s) acc[s][0] = acc[s][1] = 0ull;
    stage(0, 0);
    for (int k0 = 0, st = 0; k0 < kFlat; k0 += kTlK, st ^= 1) {
        if (k0 + kTlK < kFlat) {
            stage(st ^ 1, k0 + kTlK);
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
        const float* f = M.f[st] + 4 * warp * kTlK;
        const __nv_bfloat16* wk = M.w[st] + 4 * lane;
        // the stage's own sums, then added: chains of 64 and 21 instead of 1286
        f32x2 part[4][2];
#pragma unroll
        for (int s = 0; s < 4; ++s) part[s][0] = part[s][1] = 0ull;
#pragma unroll 4
        for (int k = 0; k < kTlK; k += 4) {
            f32x2 wa[4], wb[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint2 r = *reinterpret_cast<const uint2*>(wk + (k + q) * kHid);
                wa[q] = bfx2(r.x), wb[q] = bfx2(r.y);
            }
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const float4 v = *reinterpret_cast<const float4*>(f + s * kTlK + k);
                const float vq[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const f32x2 vv = pack2(vq[q], vq[q]);
                    part[s][0] = fma2(wa[q], vv, part[s][0]);
                    part[s][1] = fma2(wb[q], vv, part[s][1]);
                }
            }
        }
        const f32x2 one = pack2(1.0f, 1.0f);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            acc[s][0] = fma2(part[s][0], one, acc[s][0]);
            acc[s][1] = fma2(part[s][1], one, acc[s][1]);
        }
        __syncthreads();
    }
    // the motion inputs, then bias and ReLU
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const int ls = 4 * warp + s, b = b0 + min(ls, nb - 1);
#pragma unroll
        for (int k = 0; k < kMotion; ++k) {
            const uint2 r = *reinterpret_cast<const uint2*>(wt + kT4 + (kFlat + k) * kHid + 4 * lane);
            const float m = mo[(size_t)b * kMotion + k];
            acc[s][0] = fma2(bfx2(r.x), pack2(m, m), acc[s][0]);
            acc[s][1] = fma2(bfx2(r.y), pack2(m, m), acc[s][1]);
        }
        const float2 a = unpack2(acc[s][0]), c = unpack2(acc[s][1]);
        const float v[4] = {a.x, a.y, c.x, c.y};
#pragma unroll
        for (int k = 0; k < 4; ++k) M.hs[ls][4 * lane + k] = fmaxf(v[k] + wv(w, kF1.b + 4 * lane + k), 0.0f);
    }
    __syncthreads();
    for (int s = 0; s < nb; ++s) fc2_sample<TRAIN>(M.hs[s], M.ys[s], w, b0 + s, B, y, t);
    if (!TRAIN) return;
    __syncthreads();
    for (int s = 0; s < nb; ++s) fc2_backward(M.hs[s], M.ys[s], w, b0 + s, B, h, dy, dh, loss_b);
}

// d3[b,i] = (sum_o fc1.w[o,i] dh[b,o]) (a3[b,i] > 0) for the 1280 conv3
// features: one feature x 8 samples per thread, 256 features per block, whose
// weights (contiguous in the transposed copy) are staged once; their rows are
// padded to 272 bytes so that the lanes' 16-byte reads meet different banks.
constexpr int kD3Threads = 256, kD3Pitch = kHid + 8;
constexpr size_t kD3Smem = (size_t)kD3Threads * kD3Pitch * sizeof(__nv_bfloat16);

__global__ void __launch_bounds__(kD3Threads)
fc1_input_grad(const float* __restrict__ dh, const __nv_bfloat16* __restrict__ wt, const float* __restrict__ a3, int B,
               float* __restrict__ d3)
{
    extern __shared__ __align__(16) __nv_bfloat16 ws[];
    __shared__ __align__(16) float d[kHid][kFcS];
    const int tid = threadIdx.x, b0 = blockIdx.x * kFcS, nb = min(kFcS, B - b0), i0 = blockIdx.y * kD3Threads;
#pragma unroll
    for (int q = 0; q < kHid / 8; ++q) {
        const int v = tid + q * kD3Threads, r = v / (kHid / 8), c = v % (kHid / 8);
        cp_async16(ws + r * kD3Pitch + 8 * c, wt + kT4 + (size_t)(i0 + r) * kHid + 8 * c);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
#pragma unroll
    for (int q = 0; q < kFcS * kHid / kD3Threads; ++q) {
        const int i = tid + q * kD3Threads, s = i / kHid, o = i % kHid;
        d[o][s] = s < nb ? dh[(size_t)b0 * kHid + i] : 0.0f;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    f32x2 acc[kFcS / 2];
#pragma unroll
    for (int s = 0; s < kFcS / 2; ++s) acc[s] = 0ull;
#pragma unroll 4
    for (int o = 0; o < kHid; o += 8) {
        const uint4 r = *reinterpret_cast<const uint4*>(ws + tid * kD3Pitch + o);
        const unsigned rw[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float wq = __uint_as_float((q & 1) ? rw[q / 2] & 0xffff0000u : rw[q / 2] << 16);
            const f32x2 ww = pack2(wq, wq);
            const ulonglong2 va = *reinterpret_cast<const ulonglong2*>(&d[o + q][0]);
            const ulonglong2 vb = *reinterpret_cast<const ulonglong2*>(&d[o + q][4]);
            acc[0] = fma2(ww, va.x, acc[0]);
            acc[1] = fma2(ww, va.y, acc[1]);
            acc[2] = fma2(ww, vb.x, acc[2]);
            acc[3] = fma2(ww, vb.y, acc[3]);
        }
    }
#pragma unroll
    for (int s = 0; s < kFcS; ++s) {
        if (s >= nb) break;
        const size_t at = (size_t)(b0 + s) * kFlat + i0 + tid;
        const float2 v = unpack2(acc[s / 2]);
        d3[at] = a3[at] > 0.0f ? ((s & 1) ? v.y : v.x) : 0.0f;
    }
}

// Weight and bias gradients of the fully connected layers: dW[o,i] = sum_b
// dz[b,o] in[b,i], the bias as one more input of ones.  A block takes 16
// inputs of fc1 and all 128 outputs (4 outputs x 2 inputs per thread), the
// samples staged 64 at a time in two stages; blocks past those take fc2's.
constexpr int kGwThreads = 256, kGwK = 64, kGwI = 16;
constexpr int kGwB1 = (kF + 1 + kGwI - 1) / kGwI, kGwB2 = (kHid + 1 + 31) / 32, kGwBlocks = kGwB1 + kGwB2;

__global__ void __launch_bounds__(kGwThreads)
fc_weight_grad(const float* __restrict__ dh, const float* __restrict__ dy, const float* __restrict__ a3,
               const float* __restrict__ mo, const float* __restrict__ h, int B, float* __restrict__ grad)
{
    extern __shared__ __align__(16) float smw[];
    const int tid = threadIdx.x;
    if (blockIdx.x >= kGwB1) {
        // fc2: 8 outputs x 32 inputs, one per thread
        const int o = tid >> 5, i = (blockIdx.x - kGwB1) * 32 + (tid & 31);
        float s = 0.0f;
#pragma unroll 8
        for (int b = 0; b < B; ++b)
            s = fmaf(dy[(size_t)b * kOut + o], i < kHid ? h[(size_t)b * kHid + i] : 1.0f, s);
        if (i <= kHid) grad[i == kHid ? kF2.b + o : kF2.w + o * kHid + i] = s;
        return;
    }
    float* zs = smw;                              // [2][kGwK][kHid]
    float* is = smw + 2 * kGwK * kHid;            // [2][kGwK][kGwI]
    const int i0 = blockIdx.x * kGwI;
    auto stage = [&](int st, int b0) {
#pragma unroll
        for (int q = 0; q < kGwK * kHid / 4 / kGwThreads; ++q) {
            const int e = tid + q * kGwThreads, b = b0 + e / (kHid / 4);
            float* to = zs + st * kGwK * kHid + 4 * e;
            if (b < B)
                cp_async16(to, dh + (size_t)b0 * kHid + 4 * e);
            else
                *reinterpret_cast<float4*>(to) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        const int r = tid / (kGwI / 4), c = 4 * (tid % (kGwI / 4)), b = b0 + r;
        float* to = is + (st * kGwK + r) * kGwI + c;
        if (b < B && i0 + c < kFlat) {
            cp_async16(to, a3 + (size_t)b * kFlat + i0 + c);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + c + q;
                to[q] = b >= B || i > kF ? 0.0f : i == kF ? 1.0f : mo[(size_t)b * kMotion + (i - kFlat)];
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    static_assert(kGwK * kGwI / 4 == kGwThreads && kFlat % kGwI == 0, "one input quad per thread");
    const int to = (tid & 31) * 4, ti = (tid >> 5) * 2;
    f32x2 acc[2][2];
#pragma unroll
    for (int q = 0; q < 2; ++q) acc[q][0] = acc[q][1] = 0ull;
    stage(0, 0);
    for (int b0 = 0, st = 0; b0 < B; b0 += kGwK, st ^= 1) {
        if (b0 + kGwK < B) {
            stage(st ^ 1, b0 + kGwK);
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
        const float* z = zs + st * kGwK * kHid + to;
        const float* v = is + st * kGwK * kGwI + ti;
#pragma unroll 8
        for (int b = 0; b < kGwK; ++b) {
            const ulonglong2 zz = *reinterpret_cast<const ulonglong2*>(z + b * kHid);
            const float2 vv = *reinterpret_cast<const float2*>(v + b * kGwI);
            const f32x2 va = pack2(vv.x, vv.x), vb = pack2(vv.y, vv.y);
            acc[0][0] = fma2(zz.x, va, acc[0][0]);
            acc[0][1] = fma2(zz.y, va, acc[0][1]);
            acc[1][0] = fma2(zz.x, vb, acc[1][0]);
            acc[1][1] = fma2(zz.y, vb, acc[1][1]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i = i0 + ti + q;
        if (i > kF) continue;
        const float2 a = unpack2(acc[q][0]), b = unpack2(acc[q][1]);
        const float v[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
        for (int k = 0; k < 4; ++k) grad[i == kF ? kF1.b + to + k : kF1.w + (to + k) * kF + i] = v[k];
    }
}

// ---------------------------------------------------------------------------
// Backward pass of the convolutions, in two kernels (together they would hold
// 80 gradient sums a thread beside the input gradients' registers and spilled as
// many; conv_weight_grad alone spills 84 bytes):
//  * conv_input_grad: d2 from d3 and d1 from d2, a sample per block at a time.
//    A thread owns a 2 x 2 quad of input pixels x 4 channels, whose nine
//    (pixel, tap) pairs use each weight once (36 FMAs per 9 + 4 shared loads);
//    the lanes of a warp take the quads of one channel group, so its weight
//    loads are broadcasts; the output channels are split over warp groups;
//  * conv_weight_grad: a block takes whole samples and carries its sums in
//    registers over all of them.  A thread owns 8 output channels x the 9 taps
//    of one input channel (72 sums; 72 FMAs per 2 + 9 shared loads): half of
//    the block conv3's, the other half conv2's with the positions split over
//    four thread groups; conv1 one (channel, row) per thread.  Input planes
//    have an odd stride, so the lanes of a warp (channels) read different
//    banks.  The blocks' sums go to `part`; adam_update adds them in order.
// Both bound by FP32 issue and the shared-memory pipe.
// ---------------------------------------------------------------------------
constexpr int kBwThreads = 512;
constexpr int kP1 = 375, kP2 = 121;                       // plane strides of a1 (17 x 22) and a2 (10 x 12)
constexpr int kD3P = 68, kD2P = 36;                       // position strides of d3 and d2 (banks staggered)
constexpr int kPart = kW3 + 64 + kW2 + 32 + 144 + 16;     // one block's sums: conv3, conv2, conv1 (w, b each)
constexpr int kPt3 = 0, kPt2 = kW3 + 64, kPt1 = kPt2 + kW2 + 32;

// Place e of a block's sums ([tap][output channel][input channel], then the
// biases, of conv3 and conv2; conv1 in file order) -> parameter.
__device__ __forceinline__ int part_param(int e)
{
    if (e >= kPt1) return e - kPt1;
    const bool third = e < kPt2;
    const int C = third ? 32 : 16, O = third ? 64 : 32, q = third ? e : e - kPt2, base = third ? kC3.w : kC2.w;
    if (q >= 9 * O * C) return base + q;                  // bias
    const int c = q % C, o = (q / C) % O, tap = q / (C * O);
    return base + (o * C + c) * 9 + tap;
}

struct IgSmem {
    float w3[kW3], w2[kW2];             // [output channel][tap][input channel]
    float d3p[64 * 30];                 // [channel][5 x 6], zero beyond 4 x 5
    float d2p[32 * 99];                 // [channel][9 x 11], zero beyond 8 x 10
    float tmp[16 * 160];                // the other warp groups' part of a gradient
};
static_assert(offsetof(IgSmem, w2) % 16 == 0, "16-byte reads");

struct WgSmem {
    float x[32 * 42], a1[16 * kP1], a2[32 * kP2];
    float d3[20 * kD3P];                // [position][channel]
    float d2[80 * kD2P];                // [position][channel]
    float d1[16 * 301];                 // [channel][15 x 20]
    float red[4 * kW2], tmp[128];
};
static_assert(offsetof(WgSmem, d3) % 16 == 0 && offsetof(WgSmem, d2) % 16 == 0, "16-byte reads");

// the quad (i0, j0) of an input gradient: acc[px][channel] over output
// channels [o0, o1); dp: padded gradient planes of stride DP and row DW;
// w: [o][tap][C]
template <int C, int DP, int DW>
__device__ __forceinline__ void quad_grad(const float* __restrict__ dp, const float* __restrict__ w, int o0, int o1,
                                          int i0, int j0, int c0, float (&acc)[4][4])
{
    f32x2 s[4][2];
#pragma unroll
    for (int p = 0; p < 4; ++p) s[p][0] = s[p][1] = 0ull;
#pragma unroll 2
    for (int o = o0; o < o1; ++o) {
        const float* d = dp + o * DP + i0 * DW + j0;
        const f32x2 d00 = pack2(d[0], d[0]), d01 = pack2(d[1], d[1]), d10 = pack2(d[DW], d[DW]),
                    d11 = pack2(d[DW + 1], d[DW + 1]);
        const float* wo = w + o * 9 * C + c0;
        // input row 2 i0 takes tap row 1 of output row i0; row 2 i0 + 1 tap row
        // 2 of i0 and tap row 0 of i0 + 1; columns alike
        auto tap = [&](int q, int px, f32x2 v) {
            const ulonglong2 r = *reinterpret_cast<const ulonglong2*>(wo + q * C);
            s[px][0] = fma2(r.x, v, s[px][0]);
            s[px][1] = fma2(r.y, v, s[px][1]);
        };
        tap(4, 0, d00);
        tap(3, 1, d01);
        tap(5, 1, d00);
        tap(1, 2, d10);
        tap(7, 2, d00);
        tap(0, 3, d11);
        tap(2, 3, d10);
        tap(6, 3, d01);
        tap(8, 3, d00);
    }
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const float2 a = unpack2(s[p][0]), b = unpack2(s[p][1]);
        acc[p][0] = a.x, acc[p][1] = a.y, acc[p][2] = b.x, acc[p][3] = b.y;
    }
}

// weight-gradient sums of 8 output channels x 9 taps of one input plane over
// positions [p0, p1)
template <int WO, int Wp, int DP>
__device__ __forceinline__ void tap_grad(const float* __restrict__ dpos, const float* __restrict__ plane, int p0, int p1,
                                         int og, f32x2 (&acc)[4][9], f32x2 (&bias)[4])
{
    const f32x2 one = pack2(1.0f, 1.0f);
    for (int p = p0; p < p1; ++p) {
        const ulonglong2 da = *reinterpret_cast<const ulonglong2*>(dpos + p * DP + og * 8);
        const ulonglong2 db = *reinterpret_cast<const ulonglong2*>(dpos + p * DP + og * 8 + 4);
        const f32x2 dv[4] = {da.x, da.y, db.x, db.y};
        const float* in = plane + 2 * (p / WO) * Wp + (p % WO);
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float v = in[(q / 3) * Wp + ((q % 3) & 1) * (Wp / 2) + ((q % 3) >> 1)];
            const f32x2 vv = pack2(v, v);
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[k][q] = fma2(dv[k], vv, acc[k][q]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) bias[k] = fma2(dv[k], one, bias[k]);
    }
}

__global__ void __launch_bounds__(kBwThreads, 1)
conv_input_grad(const float* __restrict__ d3, const float* __restrict__ a1, const float* __restrict__ a2,
                const __nv_bfloat16* __restrict__ wt, int B, float* __restrict__ d2, float* __restrict__ d1)
{
    extern __shared__ __align__(16) unsigned char raw[];
    IgSmem& M = *reinterpret_cast<IgSmem*>(raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // BF16 weights, 8 at a time: conv2's part, then conv3's
    static_assert(kB3 == kB2 + kW2, "one contiguous copy");
#pragma unroll
    for (int q = 0; q < ((kW2 + kW3) / 8 + kBwThreads - 1) / kBwThreads; ++q) {
        const int e = 8 * (tid + q * kBwThreads);
        if (e < kW2 + kW3) {
            const uint4 r = *reinterpret_cast<const uint4*>(wt + kB2 + e);
            float* to = e < kW2 ? M.w2 + e : M.w3 + e - kW2;
            const float2 a = bf2(r.x), b = bf2(r.y), c = bf2(r.z), d = bf2(r.w);
            *reinterpret_cast<float4*>(to) = make_float4(a.x, a.y, b.x, b.y);
            *reinterpret_cast<float4*>(to + 4) = make_float4(c.x, c.y, d.x, d.y);
        }
    }
    for (int i = tid; i < 64 * 30 + 32 * 99; i += kBwThreads) M.d3p[i] = 0.0f;
    __syncthreads();
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int i = tid + q * kBwThreads, o = i / 20, p = i % 20;
            if (i < kFlat) M.d3p[o * 30 + (p / 5) * 6 + p % 5] = d3[(size_t)b * kFlat + i];
        }
        __syncthreads();
        // d2: warp = half of conv3's channels x channel group of 4, lanes 0-19 the quads
        {
            const int half = warp >> 3, cg = warp & 7, e = cg * 20 + lane;
            const bool on = lane < 20;
            const int i0 = on ? lane / 5 : 0, j0 = on ? lane % 5 : 0;
            float acc[4][4], m[4][4];
            if (on && half == 0) {
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        m[p][k] = a2[((size_t)b * 32 + cg * 4 + k) * 80 + (2 * i0 + (p >> 1)) * 10 + 2 * j0 + (p & 1)];
            }
            quad_grad<32, 30, 6>(M.d3p, M.w3, half * 32, half * 32 + 32, i0, j0, cg * 4, acc);
            if (on && half == 1) {
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int k = 0; k < 4; ++k) M.tmp[(p * 4 + k) * 160 + e] = acc[p][k];
            }
            __syncthreads();
            if (on && half == 0) {
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const int yy = 2 * i0 + (p >> 1), xx = 2 * j0 + (p & 1);
                    float v[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        v[k] = m[p][k] > 0.0f ? acc[p][k] + M.tmp[(p * 4 + k) * 160 + e] : 0.0f;
                        M.d2p[(cg * 4 + k) * 99 + yy * 11 + xx] = v[k];
                    }
                    *reinterpret_cast<float4*>(d2 + ((size_t)b * 80 + yy * 10 + xx) * 32 + cg * 4) =
                        make_float4(v[0], v[1], v[2], v[3]);
                }
            }
            __syncthreads();
        }
        // d1: warps 0-11, 3 per channel group of 4
        {
            const int cg = warp / 3, quad = (warp % 3) * 32 + lane;
            if (cg < 4 && quad < 80) {
                const int i0 = quad / 10, j0 = quad % 10;
                float acc[4][4];
                quad_grad<16, 99, 11>(M.d2p, M.w2, 0, 32, i0, j0, cg * 4, acc);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const int yy = 2 * i0 + (p >> 1), xx = 2 * j0 + (p & 1);
                    if (yy >= 15) continue;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const size_t at = ((size_t)b * 16 + cg * 4 + k) * 300 + yy * 20 + xx;
                        d1[at] = a1[at] > 0.0f ? acc[p][k] : 0.0f;
                    }
                }
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kBwThreads, 1)
conv_weight_grad(const float* __restrict__ x, const float* __restrict__ a1, const float* __restrict__ a2,
                 const float* __restrict__ d3, const float* __restrict__ d2, const float* __restrict__ d1, int B,
                 float* __restrict__ part)
{
    extern __shared__ __align__(16) unsigned char raw[];
    WgSmem& M = *reinterpret_cast<WgSmem*>(raw);
    const int tid = threadIdx.x;
    for (int i = tid; i < 32 * 42 + 16 * kP1 + 32 * kP2; i += kBwThreads) M.x[i] = 0.0f;
    // weight-gradient roles: threads 0-255 conv3 (8 output groups x 32 input
    // channels), the others conv2 (4 position groups x 4 x 16)
    const bool third = tid < 256;
    const int u = tid & 255, gc = third ? u & 31 : u & 15, gg = third ? u >> 5 : (u >> 4) & 3, gs = u >> 6;
    const int o1 = tid & 15, r1 = tid >> 4;               // conv1: channel, row (r1 < 15)
    f32x2 wg[4][9], bg[4];
    float w1g[9], b1g = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        bg[k] = 0ull;
#pragma unroll
        for (int q = 0; q < 9; ++q) wg[k][q] = 0ull;
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) w1g[q] = 0.0f;
    __syncthreads();
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
#pragma unroll 5
        for (int q = 0; q < 10; ++q) {
            const int i = tid + q * kBwThreads;
            if (i < 4800) {
                const float va = a1[(size_t)b * 4800 + i], vd = d1[(size_t)b * 4800 + i];
                const int c = i / 300, p = i % 300;
                M.a1[c * kP1 + (p / 20 + 1) * 22 + split_col(p % 20 + 1, 22)] = va;
                M.d1[c * 301 + p] = vd;
            }
        }
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            const int i = tid + q * kBwThreads, c = i / 80, p = i % 80;
            const float va = a2[(size_t)b * 2560 + i], vd = d2[(size_t)b * 2560 + i];
            M.a2[c * kP2 + (p / 10 + 1) * 12 + split_col(p % 10 + 1, 12)] = va;
            M.d2[(i >> 5) * kD2P + (i & 31)] = vd;
            if (q < 3) {
                if (i < kIn) M.x[(i / 40 + 1) * 42 + split_col(i % 40 + 1, 42)] = x[(size_t)b * kIn + i];
                if (i < kFlat) M.d3[(i % 20) * kD3P + i / 20] = d3[(size_t)b * kFlat + i];
            }
        }
        __syncthreads();
        if (third)
            tap_grad<5, 12, kD3P>(M.d3, M.a2 + gc * kP2, 0, 20, gg, wg, bg);
        else
            tap_grad<10, 22, kD2P>(M.d2, M.a1 + gc * kP1, gs * 20, gs * 20 + 20, gg, wg, bg);
        if (r1 < 15) {
            const float* d = M.d1 + o1 * 301 + r1 * 20;
            const float* in = M.x + 2 * r1 * 42;
            for (int j = 0; j < 20; ++j) {
                const float dv = d[j];
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    w1g[q] = fmaf(dv, in[(q / 3) * 42 + ((q % 3) & 1) * 21 + ((q % 3) >> 1) + j], w1g[q]);
                b1g += dv;
            }
        }
        __syncthreads();
    }
    // this block's sums: conv2's position groups and conv1's rows meet in
    // shared memory, in order
    float* out = part + (size_t)blockIdx.x * kPart;
    float* red = M.red;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int o = gg * 8 + 2 * k;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float2 v = unpack2(wg[k][q]);
            float* to = third ? out + kPt3 + (q * 64 + o) * 32 + gc : red + gs * kW2 + (q * 32 + o) * 16 + gc;
            to[0] = v.x;
            to[third ? 32 : 16] = v.y;
        }
        if (gc == 0) {
            const float2 v = unpack2(bg[k]);
            float* to = third ? out + kPt3 + kW3 + o : M.tmp + gs * 32 + o;
            to[0] = v.x;
            to[1] = v.y;
        }
    }
    if (r1 < 15) {
#pragma unroll
        for (int q = 0; q < 9; ++q) M.d1[r1 * 160 + o1 * 9 + q] = w1g[q];
        M.d1[r1 * 160 + 144 + o1] = b1g;
    }
    __syncthreads();
    for (int i = tid; i < kW2; i += kBwThreads) out[kPt2 + i] = ((red[i] + red[kW2 + i]) + red[2 * kW2 + i]) + red[3 * kW2 + i];
    if (tid < 32) out[kPt2 + kW2 + tid] = ((M.tmp[tid] + M.tmp[32 + tid]) + M.tmp[64 + tid]) + M.tmp[96 + tid];
    if (tid < 160) {
        float s = 0.0f;
        for (int r = 0; r < 15; ++r) s += M.d1[r * 160 + tid];
        out[kPt1 + tid] = s;
    }
}

// Gradient of every parameter (the convolutions' from the blocks' sums, in
// block order over four interleaved quarters, with the additions' rounding
// errors kept) and, with ADAM, the update (Kingma and Ba) of the FP32 master
// weights and the BF16 copies.  Blocks below kAdConv take 64 convolution
// parameters each, four threads per parameter; the rest 256 parameters of the
// fully connected layers; the last one adds the loss terms.  Without the
// rounding errors (chains of 37 additions) conv3's gradient had 1.06 to 1.11
// times the error against 64 bits of 128 chains and a tree over all terms, at
// 148 to 256 samples; with them 0.68 to 0.88 times, and no layer's is larger.
constexpr int kAdConvN = kPart, kAdConv = (kAdConvN + 63) / 64;
constexpr int kAdFc = (kParams - kF1.w + 255) / 256, kAdBlocks = kAdConv + kAdFc + 1;
static_assert(kAdConvN == kF1.w, "the convolutions' parameters come first");

// s.x + s.y += v, with the rounding of s.x + v kept in s.y (TwoSum, Knuth)
__device__ __forceinline__ void add_exact(float2& s, float v)
{
    const float t = s.x + v, z = t - s.x;
    s.y += (s.x - (t - z)) + (v - z);
    s.x = t;
}

template <bool ADAM>
__global__ void __launch_bounds__(256)
adam_update(float* __restrict__ w, __nv_bfloat16* __restrict__ wbf, __nv_bfloat16* __restrict__ wt,
            float* __restrict__ g, const float* __restrict__ part, int nparts, float* __restrict__ m,
            float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2,
            const float* __restrict__ loss_b, int B, float* __restrict__ loss)
{
    int i = -1;
    float gi = 0.0f;
    if (blockIdx.x < kAdConv) {
        __shared__ float2 q4[4][64];
        const int e = threadIdx.x & 63, q = threadIdx.x >> 6, at = blockIdx.x * 64 + e;
        float2 s = make_float2(0.0f, 0.0f);
        if (at < kAdConvN) {
#pragma unroll 8
            for (int k = q; k < nparts; k += 4) add_exact(s, part[(size_t)k * kPart + at]);
        }
        q4[q][e] = s;
        __syncthreads();
        if (q == 0 && at < kAdConvN) {
            i = part_param(at);
            float lo = s.y;
#pragma unroll
            for (int r = 1; r < 4; ++r) {
                s.y = 0.0f;
                add_exact(s, q4[r][e].x);
                lo += q4[r][e].y + s.y;
            }
            gi = isfinite(s.x) ? s.x + lo : s.x;
            g[i] = gi;
        }
    } else if (blockIdx.x < kAdConv + kAdFc) {
        const int c = kF1.w + (blockIdx.x - kAdConv) * 256 + threadIdx.x;
        if (c < kParams) {
            i = c;
            gi = g[i];
        }
    } else {
        // loss = 0.5 / B sum_b |y_b - t_b|^2
        __shared__ float red[256];
        float s = 0.0f;
        for (int b = threadIdx.x; b < B; b += 256) s += loss_b[b];
        red[threadIdx.x] = s;
        __syncthreads();
        for (int st = 128; st > 0; st >>= 1) {
            if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
            __syncthreads();
        }
        if (threadIdx.x == 0) *loss = 0.5f * red[0] / (float)B;
    }
    if (!ADAM || i < 0) return;
    const float mi = fmaf(b1, m[i], (1.0f - b1) * gi);
    const float vi = fmaf(b2, v[i], (1.0f - b2) * gi * gi);
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    w[i] = wi;
    const __nv_bfloat16 wb = __float2bfloat16_rn(wi);
    wbf[i] = wb;
    put_wt(wt, i, wb);
}

// The BF16 copies of the master weights (after a change from the host).
__global__ void to_bf16(const float* __restrict__ w, __nv_bfloat16* __restrict__ wbf, __nv_bfloat16* __restrict__ wt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kParams) return;
    const __nv_bfloat16 b = __float2bfloat16_rn(w[i]);
    wbf[i] = b;
    put_wt(wt, i, b);
}

}  // namespace nn
}  // namespace glt

struct glt_nn {
    int max_batch = 0;
    int step = 0;
    int sms = 0;                      // multiprocessors of the device
    float* w = nullptr;               // FP32 master
    __nv_bfloat16* wbf = nullptr;     // BF16 copy used by the kernels
    __nv_bfloat16* wt = nullptr;      // the same weights relayouted (kT2 ..)
    float* g = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    // activations and gradients of up to max_batch samples, the backward
    // blocks' weight-gradient sums, loss terms
    float *a1 = nullptr, *a2 = nullptr, *a3 = nullptr, *h = nullptr, *y = nullptr, *dy = nullptr, *dh = nullptr,
          *d3 = nullptr, *d2 = nullptr, *d1 = nullptr, *part = nullptr, *loss_b = nullptr;
    float* loss = nullptr;
};

using namespace glt;
using namespace glt::nn;

namespace {

constexpr size_t kGwSmem = (size_t)2 * kGwK * (kHid + kGwI) * sizeof(float);
// fc_forward_split up to this many samples, fc_forward_tile beyond.  Split against
// tile: 512 samples forward 48 / 74 us, 1536 115 / 119, 2048 148 / 142, 4096 264 /
// 214; a training step of 1536 495 / 514 us, 2048 651 / 658, 2560 807 / 803.
constexpr int kFcSmall = 2048;

int nn_alloc(glt_nn* n)
{
    const int B = n->max_batch;
    auto al = [](float** p, size_t count) {
        return cudaMalloc(reinterpret_cast<void**>(p), count * sizeof(float));
    };
    cudaError_t e = cudaSuccess;
    int dev = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = al(&n->w, kParams);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->wbf), kParams * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->wt), kWt * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = al(&n->g, kParams);
    if (e == cudaSuccess) e = al(&n->m, kParams);
    if (e == cudaSuccess) e = al(&n->v, kParams);
    if (e == cudaSuccess) e = al(&n->a1, (size_t)B * 16 * 15 * 20);
    if (e == cudaSuccess) e = al(&n->a2, (size_t)B * 32 * 8 * 10);
    if (e == cudaSuccess) e = al(&n->a3, (size_t)B * kFlat);
    if (e == cudaSuccess) e = al(&n->h, (size_t)B * kHid);
    if (e == cudaSuccess) e = al(&n->y, (size_t)B * kOut);
    if (e == cudaSuccess) e = al(&n->dy, (size_t)B * kOut);
    if (e == cudaSuccess) e = al(&n->dh, (size_t)B * kHid);
    if (e == cudaSuccess) e = al(&n->d3, (size_t)B * kFlat);
    if (e == cudaSuccess) e = al(&n->d2, (size_t)B * 32 * 8 * 10);
    if (e == cudaSuccess) e = al(&n->d1, (size_t)B * 16 * 15 * 20);
    if (e == cudaSuccess) e = al(&n->part, (size_t)std::min(B, n->sms) * kPart);
    if (e == cudaSuccess) e = al(&n->loss_b, (size_t)B);
    if (e == cudaSuccess) e = al(&n->loss, 1);
    if (e == cudaSuccess) e = cudaMemset(n->m, 0, kParams * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(n->v, 0, kParams * sizeof(float));
    auto smem = [](auto k, size_t bytes) {
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    if (e == cudaSuccess) e = smem(conv_forward<2, false>, sizeof(FwdSmem<2>));
    if (e == cudaSuccess) e = smem(conv_forward<2, true>, sizeof(FwdSmem<2>));
    if (e == cudaSuccess) e = smem(conv_forward<4, false>, sizeof(FwdSmem<4>));
    if (e == cudaSuccess) e = smem(conv_forward<4, true>, sizeof(FwdSmem<4>));
    if (e == cudaSuccess) e = smem(fc_forward_split<false>, sizeof(SplitSmem));
    if (e == cudaSuccess) e = smem(fc_forward_split<true>, sizeof(SplitSmem));
    if (e == cudaSuccess) e = smem(fc_forward_tile<false>, sizeof(TileSmem));
    if (e == cudaSuccess) e = smem(fc_forward_tile<true>, sizeof(TileSmem));
    if (e == cudaSuccess) e = smem(fc1_input_grad, kD3Smem);
    if (e == cudaSuccess) e = smem(fc_weight_grad, kGwSmem);
    if (e == cudaSuccess) e = smem(conv_input_grad, sizeof(IgSmem));
    if (e == cudaSuccess) e = smem(conv_weight_grad, sizeof(WgSmem));
    return e == cudaSuccess ? GLT_OK : cuda_fail(e, "proposal network allocation");
}

void nn_free(glt_nn* n)
{
    if (!n) return;
    for (float* p : {n->w, n->g, n->m, n->v, n->a1, n->a2, n->a3, n->h, n->y, n->dy, n->dh, n->d3, n->d2, n->d1, n->part, n->loss_b,
                     n->loss})
        cudaFree(p);
    cudaFree(n->wbf);
    cudaFree(n->wt);
    delete n;
}

int grid_for(int n, int t) { return (n + t - 1) / t; }

// Blocks of the convolutions' backward kernels, and so of the sums in `part`: one
// per multiprocessor, each of whole samples.  148 on this part's 152 left four
// idle and cost a round where B just passes a multiple: 149 samples 113 instead of
// 93 us a training step, 304 148 instead of 128, 256 the same.
int bw_blocks(const glt_nn* n, int B) { return std::min(B, n->sms); }

// conv1-conv3 of B samples; TRAIN: the activations are kept
template <bool TRAIN>
void launch_conv_forward(const glt_nn* n, const float* x, int B, cudaStream_t s)
{
    if (grid_for(B, kFwdSmall) <= n->sms)
        conv_forward<2, TRAIN><<<grid_for(B, 2), kFwdThreads, sizeof(FwdSmem<2>), s>>>(x, n->wbf, n->wt, B, n->a1, n->a2, n->a3);
    else
        conv_forward<4, TRAIN><<<std::min(grid_for(B, 4), n->sms), kFwdThreads, sizeof(FwdSmem<4>), s>>>(
            x, n->wbf, n->wt, B, n->a1, n->a2, n->a3);
}

// fc1 and fc2 of B samples; TRAIN: up to dh
template <bool TRAIN>
cudaError_t launch_fc_forward(const glt_nn* n, const float* mo, int B, float* y, const float* t, cudaStream_t s)
{
    if (B > kFcSmall) {
        fc_forward_tile<TRAIN><<<grid_for(B, kTlS), kTlThreads, sizeof(TileSmem), s>>>(n->a3, mo, n->wbf, n->wt, B, y, t, n->h,
                                                                                      n->dy, n->dh, n->loss_b);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(grid_for(B, kFcS) * kSpC), 1, 1);
    cfg.blockDim = dim3(kSpThreads, 1, 1);
    cfg.dynamicSmemBytes = sizeof(SplitSmem);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kSpC;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fc_forward_split<TRAIN>, (const float*)n->a3, mo, (const __nv_bfloat16*)n->wbf,
                              (const __nv_bfloat16*)n->wt, B, y, t, n->h, n->dy, n->dh, n->loss_b);
}

// The status of a call's launches so far: `e`, that of the last one, or the
// error an earlier `<<<>>>` left (none is left for a later call either way).
cudaError_t launches_status(cudaError_t e)
{
    const cudaError_t earlier = cudaGetLastError();
    return e != cudaSuccess ? e : earlier;
}

cudaError_t nn_forward(const glt_nn* n, const float* x, const float* mo, int B, float* y, cudaStream_t s)
{
    launch_conv_forward<false>(n, x, B, s);
    return launches_status(launch_fc_forward<false>(n, mo, B, y, nullptr, s));
}

// forward and backward: the gradient sums up to adam_update, which completes them
cudaError_t nn_backward(const glt_nn* n, const float* x, const float* mo, const float* t, int B, cudaStream_t s)
{
    launch_conv_forward<true>(n, x, B, s);
    const cudaError_t e = launches_status(launch_fc_forward<true>(n, mo, B, n->y, t, s));
    if (e != cudaSuccess) return e;
    fc1_input_grad<<<dim3(grid_for(B, kFcS), kFlat / kD3Threads), kD3Threads, kD3Smem, s>>>(n->dh, n->wt, n->a3, B, n->d3);
    fc_weight_grad<<<kGwBlocks, kGwThreads, kGwSmem, s>>>(n->dh, n->dy, n->a3, mo, n->h, B, n->g);
    conv_input_grad<<<bw_blocks(n, B), kBwThreads, sizeof(IgSmem), s>>>(n->d3, n->a1, n->a2, n->wt, B, n->d2, n->d1);
    conv_weight_grad<<<bw_blocks(n, B), kBwThreads, sizeof(WgSmem), s>>>(x, n->a1, n->a2, n->d3, n->d2, n->d1, B, n->part);
    return cudaGetLastError();
}

bool unaligned(const float* p) { return (reinterpret_cast<uintptr_t>(p) & (alignof(float) - 1)) != 0; }

int check_batch(const glt_nn* n, int B)
{
    if (!n) return invalid_arg_msg("network is NULL");
    if (B < 1 || B > n->max_batch) return invalid_arg_msg("batch size outside [1, max_batch]");
    return GLT_OK;
}

}  // namespace

int glt::invalid_arg_msg(const char* msg)
{
    set_error(msg);
    return GLT_ERR_INVALID_ARG;
}

// ---------------------------------------------------------------------------
// Proposal stage of the batched tracker
// ---------------------------------------------------------------------------
namespace glt {
namespace nn {

// Proposal stage: one thread block per stream runs the whole inference with
// the activations in shared memory and the BF16 weights read through the
// read-only cache (they stay L2-resident across blocks):
//   x = (I_cur - I_ref) / 64 on the 40 x 30 coarsest level,
//   conv1 -> conv2 -> conv3 (ReLU) -> fc1 (ReLU) on [flatten, motion] -> fc2,
//   then T' = T exp(0.01 y[0:6]), a' = a + 0.01 y[6], b' = b + y[7].
// Conv inputs are stored with a one-pixel zero border, so every 3x3 window is
// read without bounds tests.  conv1 gives each thread 4 output channels of one
// pixel; conv2 and conv3 run as small GEMMs (output pixels x channels, K =
// input channel x tap) with register tiles of PT pixels x 4 channels, on the
// layer's weights in the [K][O] layout (a tile's 4 weights are one 8-byte
// load), copied into shared memory with asynchronous 16-byte copies issued at
// the start and awaited just before conv2.  The sum order per output is bias,
// then channel, row, column; conv_forward adds conv3 in two halves of its input
// channels and fc1 in other parts, so the two round differently.
constexpr int kPropThreads = 512;
constexpr int kXp = 32 * 42, kA1p = 16 * 17 * 22, kA2p = 32 * 10 * 12;
constexpr int kPropSmemFloats = kXp + kA1p + kA2p + (kF + 2) + kHid + kOut;
constexpr size_t kPropSmemBytes = kPropSmemFloats * sizeof(float) + (kW2 + kW3) * sizeof(__nv_bfloat16);
static_assert(kPropSmemFloats % 4 == 0, "the BF16 weights must start on a 16-byte boundary");
static_assert((kXp + kA1p + kA2p) % 4 == 0, "the bordered planes are cleared as float4");
static_assert((kW2 + kW3) * sizeof(__nv_bfloat16) % 16 == 0, "the weight copy is made of 16-byte pieces");

// GEMM form of a stride-2 3x3 conv on a zero-bordered, column-split input:
// thread t < tasks computes PT output pixels p = pg + u PG (consecutive
// lanes, consecutive pixels) x 4 channels.  Output planes bordered and
// column-split if PADOUT, else flat.
template <int C, int H, int W, int O, int PT, bool PADOUT>
__device__ __forceinline__ void conv_gemm(const float* __restrict__ in, const __nv_bfloat16* __restrict__ wt,
                                          const __nv_bfloat16* __restrict__ w, int boff,
                                          float* __restrict__ out)
{
    constexpr int Ho = (H + 1) / 2, Wo = (W + 1) / 2, Wp = W + 2, plane = (H + 2) * (W + 2), half = Wp / 2;
    constexpr int PG = Ho * Wo / PT, tasks = PG * (O / 4);
    static_assert(Ho * Wo % PT == 0, "pixel tiles must cover the output");
    static_assert(tasks <= kPropThreads, "one tile per thread");
    static_assert(Wp % 2 == 0, "column-split rows need an even padded width");
    const int t = threadIdx.x;
    if (t >= tasks) return;
    const int pg = t % PG, cg = t / PG;
    int base[PT];
#pragma unroll
    for (int u = 0; u < PT; ++u) {
        const int p = pg + u * PG;
        base[u] = 2 * (p / Wo) * Wp + (p % Wo);     // window row 2i, split column of 2j
    }
    float acc[PT][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float b = __bfloat162float(__ldg(w + boff + cg * 4 + k));
#pragma unroll
        for (int u = 0; u < PT; ++u) acc[u][k] = b;
    }
    for (int c = 0; c < C; ++c) {
        const float* xc = in + c * plane;
        const __nv_bfloat16* wc = wt + (c * 9) * O + cg * 4;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const uint2 raw = *reinterpret_cast<const uint2*>(wc + q * O);
            const float2 w01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
            const float2 w23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
            const int di = q / 3, dj = q % 3;
            const int off = di * Wp + (dj & 1) * half + (dj >> 1);   // column 2j + dj
#pragma unroll
            for (int u = 0; u < PT; ++u) {
                const float a = xc[base[u] + off];
                acc[u][0] = fmaf(w01.x, a, acc[u][0]);
                acc[u][1] = fmaf(w01.y, a, acc[u][1]);
                acc[u][2] = fmaf(w23.x, a, acc[u][2]);
                acc[u][3] = fmaf(w23.y, a, acc[u][3]);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < PT; ++u) {
        const int p = pg + u * PG, i = p / Wo, j = p % Wo;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int o = cg * 4 + k;
            const float r = fmaxf(acc[u][k], 0.0f);
            if (PADOUT)
                out[o * (Ho + 2) * (Wo + 2) + (i + 1) * (Wo + 2) + split_col(j + 1, Wo + 2)] = r;
            else
                out[(o * Ho + i) * Wo + j] = r;
        }
    }
}

__device__ __forceinline__ float2 wv2(const __nv_bfloat16* w, int i)
{
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(w + i));
}

// in: C planes of (H+2) x (W+2) with a zero border, rows column-split; out: O
// planes of the (H+1)/2 x (W+1)/2 result, bordered and column-split if
// PADOUT, else flat.
template <int C, int H, int W, int O, int KO, bool PADOUT>
__device__ __forceinline__ void conv_block(const float* __restrict__ in, const __nv_bfloat16* __restrict__ w,
                                           int woff, int boff, float* __restrict__ out)
{
    constexpr int Ho = (H + 1) / 2, Wo = (W + 1) / 2, Wp = W + 2, plane = (H + 2) * (W + 2);
    constexpr int tasks = (O / KO) * Ho * Wo;
    for (int t = threadIdx.x; t < tasks; t += kPropThreads) {
        const int p = t % (Ho * Wo), og = t / (Ho * Wo);
        const int i = p / Wo, j = p % Wo;
        float acc[KO];
#pragma unroll
        for (int k = 0; k < KO; ++k) acc[k] = __bfloat162float(__ldg(w + boff + og * KO + k));
        const float* xb = in + (2 * i) * Wp + j;      // column-split rows: column 2j + dj
        for (int c = 0; c < C; ++c) {
            float v[9];
#pragma unroll
            for (int di = 0; di < 3; ++di)
#pragma unroll
                for (int dj = 0; dj < 3; ++dj)
                    v[di * 3 + dj] = xb[c * plane + di * Wp + (dj & 1) * (Wp >> 1) + (dj >> 1)];
#pragma unroll
            for (int k = 0; k < KO; ++k) {
                const __nv_bfloat16* wk = w + woff + ((og * KO + k) * C + c) * 9;
#pragma unroll
                for (int q = 0; q < 9; ++q) acc[k] = fmaf(__bfloat162float(__ldg(wk + q)), v[q], acc[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < KO; ++k) {
            const int o = og * KO + k;
            const float r = fmaxf(acc[k], 0.0f);
            if (PADOUT)
                out[o * (Ho + 2) * (Wo + 2) + (i + 1) * (Wo + 2) + split_col(j + 1, Wo + 2)] = r;
            else
                out[(o * Ho + i) * Wo + j] = r;
        }
    }
}

// Network motion input from the stream's last inter-frame motion M = [R | t]
// (row-major 3x4): log(M) / 0.02 as (upsilon, omega).  The input is FP32, and
// so is this evaluation after the differences of M's entries it starts from
// (vee(R - R^T), trace R - 1 and, near pi, the symmetric part), which are
// formed in FP64.  sin th = |vee| / 2 and cos th = (trace - 1) / 2, th their
// atan2; omega = th / (2 sin th) vee (its series below th = 1e-4; near pi the
// axis comes from the symmetric part instead); upsilon = V^-1 t with
// V^-1 = I - W/2 + k W^2, k = (1 - A / (2 B)) / th^2, A = sin th / th,
// B = (1 - cos th) / th^2, taken below th = 0.5 as its series
// k = sum_n |B_2n| th^(2n-2) / (2n)! (Bernoulli numbers), to th^8.
constexpr float kMotionScale = 0.02f;

__device__ void motion_feature(const double* __restrict__ M, float* __restrict__ f6)
{
    const float vee[3] = {(float)(M[9] - M[6]), (float)(M[2] - M[8]), (float)(M[4] - M[1])};
    const float t[3] = {(float)M[3], (float)M[7], (float)M[11]};
    const float sn = 0.5f * sqrtf(vee[0] * vee[0] + vee[1] * vee[1] + vee[2] * vee[2]);
    const float cs = (float)(0.5 * (M[0] + M[5] + M[10] - 1.0));
    const float th = atan2f(sn, cs);
    const float pi = 3.14159265358979f;
    float w[3];
    if (th < 1e-4f) {
        const float k = 0.5f * (1.0f + th * th / 6.0f);
        for (int i = 0; i < 3; ++i) w[i] = k * vee[i];
    } else if (th < pi - 1e-4f) {
        const float k = th / (2.0f * sn);
        for (int i = 0; i < 3; ++i) w[i] = k * vee[i];
    } else {
        const double Rd[3] = {M[0], M[5], M[10]};
        int m = 0;
        for (int i = 1; i < 3; ++i)
            if (Rd[i] > Rd[m]) m = i;
        const float d = sqrtf((float)(0.5 * (Rd[m] + 1.0)));
        float a[3];
        for (int i = 0; i < 3; ++i)
            a[i] = i == m ? d : (float)(0.5 * (M[4 * i + m] + M[4 * m + i])) / (2.0f * d);
        const float na = sqrtf(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
        const float sg = (a[0] * vee[0] + a[1] * vee[1] + a[2] * vee[2]) < 0.0f ? -1.0f : 1.0f;
        for (int i = 0; i < 3; ++i) w[i] = sg * th * a[i] / na;
    }
    const float th2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    float k;
    if (th < 0.5f) {
        k = 1.0f / 12.0f + th2 * (1.0f / 720.0f + th2 * (1.0f / 30240.0f +
                                 th2 * (1.0f / 1209600.0f + th2 * (1.0f / 47900160.0f))));
    } else {
        const float sh = sinf(0.5f * th);
        const float A = sinf(th) / th, B = 2.0f * sh * sh / th2;
        k = (1.0f - A / (2.0f * B)) / th2;
    }
    // W = [w]x;  V^-1 t = t - (w x t) / 2 + k w x (w x t)
    const float wt[3] = {w[1] * t[2] - w[2] * t[1], w[2] * t[0] - w[0] * t[2], w[0] * t[1] - w[1] * t[0]};
    const float wwt[3] = {w[1] * wt[2] - w[2] * wt[1], w[2] * wt[0] - w[0] * wt[2],
                          w[0] * wt[1] - w[1] * wt[0]};
    for (int i = 0; i < 3; ++i) {
        f6[i] = (t[i] - 0.5f * wt[i] + k * wwt[i]) / kMotionScale;
        f6[3 + i] = w[i] / kMotionScale;
    }
}

// fc1 is shared by the kPropCluster blocks of a thread-block cluster (one
// stream each; blocks past the last stream only help): block r computes
// hidden units [r kHid / kPropCluster, (r + 1) kHid / kPropCluster) for every
// stream of its cluster, from the streams' feature vectors copied out of the
// peers' shared memory, and writes each result into its stream's block, so
// the 329 KB of fc1 weights are read from L2 once per cluster instead of once
// per stream.  Each output keeps its lane split and reduction order.
constexpr int kPropCluster = 4;
static_assert(kHid % (kPropCluster * (kPropThreads / 32)) == 0, "whole rows per warp");
static_assert(kPropCluster * (kF + 2) <= kA1p, "the peers' feature vectors fit where conv1's output was");

__global__ void __launch_bounds__(kPropThreads)
proposal_kernel(const PropJob* __restrict__ jobs, const double* __restrict__ motion,
                const double* __restrict__ init, const __nv_bfloat16* __restrict__ w,
                const __nv_bfloat16* __restrict__ wt, double* __restrict__ out, int S)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) float sm[];
    float* xp = sm;
    float* a1 = xp + kXp;
    float* a2 = a1 + kA1p;
    float* f = a2 + kA2p;
    float* h = f + (kF + 2);
    float* y = h + kHid;
    __nv_bfloat16* w2t = reinterpret_cast<__nv_bfloat16*>(y + kOut);
    __nv_bfloat16* w3t = w2t + kW2;
    const int s = blockIdx.x;
    const bool valid = s < S;      // block-uniform: blocks past the last stream only share fc1
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // conv2 / conv3 weights: one contiguous [K][O] copy, in flight until conv2
    for (int v = tid; v < (kW2 + kW3) / 8; v += kPropThreads) cp_async16(w2t + 8 * v, wt + kT2 + 8 * v);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    // the rows of T each lane of warp 0 composes at the end (lanes 12, 13: a, b)
    double Tr[4] = {0.0, 0.0, 0.0, 0.0};
    if (valid && warp == 0 && lane < 14) {
        const double* T = init + 14 * s;
        if (lane < 12) {
            for (int k = 0; k < 4; ++k) Tr[k] = T[4 * (lane >> 2) + k];
        } else {
            Tr[0] = T[lane];
        }
    }
    float4* z4 = reinterpret_cast<float4*>(sm);
    for (int q = tid; q < (kXp + kA1p + kA2p) / 4; q += kPropThreads) z4[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    __syncthreads();
    if (valid) {
        const PropJob J = jobs[s];
        for (int p = tid; p < kIn; p += kPropThreads) {
            const int r = p / 40, c = p % 40;
            xp[(r + 1) * 42 + split_col(c + 1, 42)] =
                ((float)J.cur[r * J.pitch + c] - (float)J.ref[r * J.pitch + c]) * (1.0f / 64.0f);
        }
        __syncthreads();
        conv_block<1, 30, 40, 16, 4, true>(xp, w, kC1.w, kC1.b, a1);
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    if (valid) {
        // the motion input, on a thread that conv2's 320 tiles leave idle
        if (tid == kPropThreads - 1) motion_feature(motion + 12 * s, f + kFlat);
        conv_gemm<16, 15, 20, 32, 2, true>(a1, w2t, w, kC2.b, a2);
        __syncthreads();
        conv_gemm<32, 8, 10, 64, 1, false>(a2, w3t, w, kC3.b, f);
    } else {
        for (int i = tid; i < kF + 2; i += kPropThreads) f[i] = 0.0f;
    }
    // every block's feature vector is complete; copy the cluster's into the
    // (dead) conv1 output area
    cluster.sync();
    float* fl = a1;
    for (int q = 0; q < kPropCluster; ++q) {
        const float* src = cluster.map_shared_rank(f, q);
        for (int i = tid; i < kF + 2; i += kPropThreads) fl[q * (kF + 2) + i] = src[i];
    }
    __syncthreads();
    // fc1: this block's kHid / kPropCluster rows for every stream of the
    // cluster, two rows per warp, BF16 pairs along the rows; each result goes
    // to its stream's block
    {
        constexpr int RPB = kHid / kPropCluster, RPW = RPB / (kPropThreads / 32);
        const int rank = (int)cluster.block_rank();
        const int o0 = rank * RPB + warp * RPW;
        float acc[RPW][kPropCluster];
#pragma unroll
        for (int k = 0; k < RPW; ++k)
#pragma unroll
            for (int q = 0; q < kPropCluster; ++q) acc[k][q] = 0.0f;
#pragma unroll 4
        for (int i = 2 * lane; i < kF; i += 64) {
            float2 fq[kPropCluster];
#pragma unroll
            for (int q = 0; q < kPropCluster; ++q) fq[q] = make_float2(fl[q * (kF + 2) + i], fl[q * (kF + 2) + i + 1]);
#pragma unroll
            for (int k = 0; k < RPW; ++k) {
                const float2 wp = wv2(w, kF1.w + (o0 + k) * kF + i);
#pragma unroll
                for (int q = 0; q < kPropCluster; ++q) {
                    acc[k][q] = fmaf(wp.x, fq[q].x, acc[k][q]);
                    acc[k][q] = fmaf(wp.y, fq[q].y, acc[k][q]);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < RPW; ++k)
#pragma unroll
            for (int q = 0; q < kPropCluster; ++q)
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) acc[k][q] += __shfl_xor_sync(0xffffffffu, acc[k][q], off);
        if (lane < RPW * kPropCluster) {
            const int k = lane / kPropCluster, q = lane % kPropCluster;
            float v = 0.0f;
#pragma unroll
            for (int kk = 0; kk < RPW; ++kk)
#pragma unroll
                for (int qq = 0; qq < kPropCluster; ++qq)
                    if (kk == k && qq == q) v = acc[kk][qq];
            cluster.map_shared_rank(h, q)[o0 + k] = fmaxf(v + wv(w, kF1.b + o0 + k), 0.0f);
        }
    }
    // every stream's hidden vector is complete (and no block reads a peer after this)
    cluster.sync();
    if (!valid) return;
    if (warp < kOut) {
        const int row = kF2.w + warp * kHid;
        float acc = 0.0f;
        for (int i = 2 * lane; i < kHid; i += 64) {
            const float2 wp = wv2(w, row + i);
            acc = fmaf(wp.x, h[i], acc);
            acc = fmaf(wp.y, h[i + 1], acc);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == 0) y[warp] = acc + wv(w, kF2.b + warp);
    }
    __syncthreads();
    if (warp != 0 || lane >= 14) return;
    // T' = T exp(d) = T + T (exp(d) - I): the increment exp(d) - I, whose
    // entries are O(|d|), in FP32 (every lane the whole 3 x 4 matrix;
    // A = sin th / th, B = (1 - cos th) / th^2, C = (th - sin th) / th^3 as
    // series below th^2 = 0.25, truncation below 1e-10 relative), the
    // composition in FP64: lane 4 r + c writes entry (r, c), lanes 12 and 13
    // the affine pair
    double* O = out + 14 * s;
    if (lane >= 12) {
        O[lane] = Tr[0] + (double)y[lane - 6] * (lane == 12 ? 0.01 : 1.0);
        return;
    }
    float d[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) d[k] = y[k] * 0.01f;
    const float w0 = d[3], w1 = d[4], w2 = d[5];
    const float th2 = w0 * w0 + w1 * w1 + w2 * w2;
    float A, B, C;
    if (th2 < 0.25f) {
        A = 1.0f - th2 * (1.0f / 6.0f - th2 * (1.0f / 120.0f - th2 * (1.0f / 5040.0f - th2 * (1.0f / 362880.0f))));
        B = 0.5f - th2 * (1.0f / 24.0f - th2 * (1.0f / 720.0f - th2 * (1.0f / 40320.0f - th2 * (1.0f / 3628800.0f))));
        C = 1.0f / 6.0f - th2 * (1.0f / 120.0f - th2 * (1.0f / 5040.0f - th2 * (1.0f / 362880.0f - th2 * (1.0f / 39916800.0f))));
    } else {
        const float th = sqrtf(th2), sn = sinf(th), sh = sinf(0.5f * th);
        A = sn / th;
        B = 2.0f * sh * sh / th2;
        C = (th - sn) / (th2 * th);
    }
    // W = [w]x, W^2 = w w^T - th^2 I; rotation increment A W + B W^2,
    // translation V t - t = B W t + C W^2 t with t = d[0:3]
    const float Wm[3][3] = {{0.0f, -w2, w1}, {w2, 0.0f, -w0}, {-w1, w0, 0.0f}};
    const float ww[3] = {w0, w1, w2};
    float dE[3][4];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float wt = 0.0f, w2t = 0.0f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float W2 = ww[k] * ww[j] - (k == j ? th2 : 0.0f);
            dE[k][j] = fmaf(A, Wm[k][j], B * W2);
            wt = fmaf(Wm[k][j], d[j], wt);
            w2t = fmaf(W2, d[j], w2t);
        }
        dE[k][3] = d[k] + fmaf(B, wt, C * w2t);
    }
    const int c = lane & 3;
    double v = c == 0 ? Tr[0] : c == 1 ? Tr[1] : c == 2 ? Tr[2] : Tr[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float e = c == 0 ? dE[k][0] : c == 1 ? dE[k][1] : c == 2 ? dE[k][2] : dE[k][3];
        v = fma(Tr[k], (double)e, v);
    }
    O[lane] = v;
}

}  // namespace nn

cudaError_t launch_proposal(glt_batch* b, const double* init_dev, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((b->S + nn::kPropCluster - 1) / nn::kPropCluster * nn::kPropCluster), 1, 1);
    cfg.blockDim = dim3(nn::kPropThreads, 1, 1);
    cfg.dynamicSmemBytes = nn::kPropSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = nn::kPropCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, nn::proposal_kernel, b->prop_jobs, b->motion_dev, init_dev,
                              (const __nv_bfloat16*)b->nn->wbf, (const __nv_bfloat16*)b->nn->wt,
                              b->prop_init, b->S);
}

}  // namespace glt

extern "C" {

int glt_batch_set_proposal(glt_batch* b, glt_nn* n, const double* motion_dev)
{
    if (!b) return invalid_arg_msg("batch is NULL");
    if (b->exec) {
        cudaGraphExecDestroy(b->exec);
        b->exec = nullptr;
    }
    if (b->graph) {
        cudaGraphDestroy(b->graph);
        b->graph = nullptr;
    }
    if (!n) {
        b->nn = nullptr;
        b->motion_dev = nullptr;
        return GLT_OK;
    }
    if (!motion_dev) return invalid_arg_msg("motion_dev is NULL");
    if (n->max_batch < b->S) return invalid_arg_msg("network max_batch is smaller than the batch");
    std::vector<PropJob> jobs(b->S);
    for (int i = 0; i < b->S; ++i) {
        glt_tracker* t = b->trk[i];
        const int l = t->L - 1;
        if (t->W[l] != 40 || t->H[l] != 30)
            return invalid_arg_msg("the proposal needs every stream's coarsest level to be 40 x 30");
        jobs[i].ref = t->pyr[GLT_REF].base + t->pyr[GLT_REF].off[l];
        jobs[i].cur = t->pyr[GLT_CUR].base + t->pyr[GLT_CUR].off[l];
        jobs[i].pitch = t->pitch[l];
    }
    cudaError_t e = cudaSuccess;
    if (!b->prop_jobs) {
        e = cudaMalloc(reinterpret_cast<void**>(&b->prop_jobs), b->S * sizeof(PropJob));
        if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&b->prop_init), (size_t)b->S * 14 * sizeof(double));
        if (e != cudaSuccess) return cuda_fail(e, "proposal buffers");
    }
    e = cudaMemcpy(b->prop_jobs, jobs.data(), b->S * sizeof(PropJob), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(nn::proposal_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)nn::kPropSmemBytes);
    if (e != cudaSuccess) return cuda_fail(e, "proposal jobs");
    b->nn = n;
    b->motion_dev = motion_dev;
    return GLT_OK;
}

int glt_nn_create(int max_batch, glt_nn** out)
{
    if (!out) return invalid_arg_msg("out is NULL");
    *out = nullptr;
    if (max_batch < 1 || max_batch > 65536) return invalid_arg_msg("max_batch must be in [1, 65536]");
    glt_nn* n = new glt_nn();
    n->max_batch = max_batch;
    int rc = nn_alloc(n);
    if (rc != GLT_OK) {
        nn_free(n);
        return rc;
    }
    *out = n;
    return GLT_OK;
}

void glt_nn_destroy(glt_nn* n) { nn_free(n); }

int glt_nn_set_params(glt_nn* n, const float* host, int count)
{
    if (!n || !host) return invalid_arg_msg("NULL argument");
    if (count != kParams) return invalid_arg_msg("count must equal GLT_NN_PARAMS");
    cudaError_t e = cudaMemcpy(n->w, host, kParams * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(n->m, 0, kParams * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(n->v, 0, kParams * sizeof(float));
    if (e != cudaSuccess) return cuda_fail(e, "glt_nn_set_params");
    to_bf16<<<grid_for(kParams, 256), 256>>>(n->w, n->wbf, n->wt);
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_fail(e, "glt_nn_set_params");
    n->step = 0;
    return GLT_OK;
}

int glt_nn_get_params(glt_nn* n, float* host, int count)
{
    if (!n || !host) return invalid_arg_msg("NULL argument");
    if (count != kParams) return invalid_arg_msg("count must equal GLT_NN_PARAMS");
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(host, n->w, kParams * sizeof(float), cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? GLT_OK : cuda_fail(e, "glt_nn_get_params");
}

int glt_nn_forward(glt_nn* n, const float* x_dev, const float* m_dev, float* y_dev, int B, void* stream)
{
    int rc = check_batch(n, B);
    if (rc != GLT_OK) return rc;
    if (!x_dev || !m_dev || !y_dev) return invalid_arg_msg("NULL argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    // an output that overlaps an input is written when all inputs have been
    // read; one that no kernel can store to (its address is no multiple of 4) by
    // a copy
    auto overlap = [&](const float* p, size_t len) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(p), b = reinterpret_cast<uintptr_t>(y_dev);
        return a < b + (size_t)B * kOut * sizeof(float) && b < a + len * sizeof(float);
    };
    const bool staged = unaligned(y_dev) || overlap(x_dev, (size_t)B * kIn) || overlap(m_dev, (size_t)B * kMotion);
    cudaError_t e = nn_forward(n, x_dev, m_dev, B, staged ? n->y : y_dev, s);
    if (e == cudaSuccess && staged)
        e = cudaMemcpyAsync(y_dev, n->y, (size_t)B * kOut * sizeof(float), cudaMemcpyDeviceToDevice, s);
    return e == cudaSuccess ? GLT_OK : cuda_fail(e, "glt_nn_forward");
}

int glt_nn_gradient(glt_nn* n, const float* x_dev, const float* m_dev, const float* t_dev, int B,
                    float* grad_host, float* loss_host, void* stream)
{
    int rc = check_batch(n, B);
    if (rc != GLT_OK) return rc;
    if (!x_dev || !m_dev || !t_dev || !grad_host) return invalid_arg_msg("NULL argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = nn_backward(n, x_dev, m_dev, t_dev, B, s);
    if (e == cudaSuccess) {
        adam_update<false><<<kAdBlocks, 256, 0, s>>>(n->w, n->wbf, n->wt, n->g, n->part, bw_blocks(n, B), n->m, n->v,
                                                     0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, n->loss_b, B, n->loss);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(grad_host, n->g, kParams * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && loss_host) e = cudaMemcpyAsync(loss_host, n->loss, sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e == cudaSuccess ? GLT_OK : cuda_fail(e, "glt_nn_gradient");
}

int glt_nn_train_step(glt_nn* n, const float* x_dev, const float* m_dev, const float* t_dev, int B,
                      float lr, float* loss_dev, void* stream)
{
    int rc = check_batch(n, B);
    if (rc != GLT_OK) return rc;
    if (!x_dev || !m_dev || !t_dev) return invalid_arg_msg("NULL argument");
    if (!(lr > 0.0f)) return invalid_arg_msg("lr must be > 0");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = nn_backward(n, x_dev, m_dev, t_dev, B, s);
    if (e != cudaSuccess) return cuda_fail(e, "glt_nn_train_step");
    n->step += 1;
    float* const loss = loss_dev && !unaligned(loss_dev) ? loss_dev : n->loss;
    const double b1 = 0.9, b2 = 0.999;
    const float c1 = (float)(1.0 / (1.0 - std::pow(b1, n->step)));
    const float c2 = (float)(1.0 / (1.0 - std::pow(b2, n->step)));
    adam_update<true><<<kAdBlocks, 256, 0, s>>>(n->w, n->wbf, n->wt, n->g, n->part, bw_blocks(n, B), n->m, n->v, lr,
                                                (float)b1, (float)b2, 1e-8f, c1, c2, n->loss_b, B, loss);
    e = cudaGetLastError();
    if (e == cudaSuccess && loss_dev && loss != loss_dev)
        e = cudaMemcpyAsync(loss_dev, loss, sizeof(float), cudaMemcpyDeviceToDevice, s);
    return e == cudaSuccess ? GLT_OK : cuda_fail(e, "glt_nn_train_step");
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Checkpoints and weight files

namespace {

const char kCkptTag[8] = {'G', 'L', 'T', 'N', 'N', 'C', 'K', '1'};

int io_fail(const char* what, const char* path)
{
    set_error(std::string(what) + ": " + (path ? path : "(null)"));
    return GLT_ERR_IO;
}

// Little-endian int32 from 4 bytes, independent of the host's byte order.
int32_t le32(const unsigned char* p)
{
    return (int32_t)((uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) |
                     ((uint32_t)p[3] << 24));
}

void put_le32(unsigned char* p, int32_t v)
{
    const uint32_t u = (uint32_t)v;
    for (int i = 0; i < 4; ++i) p[i] = (unsigned char)(u >> (8 * i));
}

bool read_floats(FILE* f, std::vector<float>& out, size_t n)
{
    std::vector<unsigned char> raw(n * 4);
    if (std::fread(raw.data(), 1, raw.size(), f) != raw.size()) return false;
    out.resize(n);
    for (size_t i = 0; i < n; ++i) {
        const uint32_t u = (uint32_t)le32(&raw[4 * i]);
        std::memcpy(&out[i], &u, 4);
    }
    return true;
}

bool write_floats(FILE* f, const std::vector<float>& v)
{
    std::vector<unsigned char> raw(v.size() * 4);
    for (size_t i = 0; i < v.size(); ++i) {
        uint32_t u;
        std::memcpy(&u, &v[i], 4);
        put_le32(&raw[4 * i], (int32_t)u);
    }
    return std::fwrite(raw.data(), 1, raw.size(), f) == raw.size();
}

// The header of a NumPy .npy file (format versions 1-3): checks that it
// describes GLT_NN_PARAMS little-endian float32 values in one C-order
// dimension and leaves `f` at the data.
int npy_header(FILE* f, const unsigned char* head8, const char* path)
{
    const int major = head8[6];
    size_t hlen = 0;
    if (major == 1) {
        unsigned char b[2];
        if (std::fread(b, 1, 2, f) != 2) return io_fail("short .npy header", path);
        hlen = (size_t)b[0] | ((size_t)b[1] << 8);
    } else if (major == 2 || major == 3) {
        unsigned char b[4];
        if (std::fread(b, 1, 4, f) != 4) return io_fail("short .npy header", path);
        hlen = (size_t)(uint32_t)le32(b);
    } else {
        return invalid_arg_msg("unsupported .npy version");
    }
    if (hlen == 0 || hlen > 65536) return invalid_arg_msg("bad .npy header length");
    std::string h(hlen, ' ');
    if (std::fread(&h[0], 1, hlen, f) != hlen) return io_fail("short .npy header", path);
    char shape[32];
    std::snprintf(shape, sizeof(shape), "(%d,)", kParams);
    if (h.find("'<f4'") == std::string::npos || h.find("'fortran_order': False") == std::string::npos ||
        h.find(shape) == std::string::npos)
        return invalid_arg_msg(".npy file is not GLT_NN_PARAMS little-endian float32 values");
    return GLT_OK;
}

}  // namespace

extern "C" {

int glt_nn_save(glt_nn* n, const char* path)
{
    if (!n || !path) return invalid_arg_msg("NULL argument");
    std::vector<float> w(kParams), m(kParams), v(kParams);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(w.data(), n->w, kParams * sizeof(float), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(m.data(), n->m, kParams * sizeof(float), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(v.data(), n->v, kParams * sizeof(float), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "glt_nn_save");
    FILE* f = std::fopen(path, "wb");
    if (!f) return io_fail("cannot open for writing", path);
    unsigned char head[16];
    std::memcpy(head, kCkptTag, 8);
    put_le32(head + 8, kParams);
    put_le32(head + 12, n->step);
    bool ok = std::fwrite(head, 1, 16, f) == 16 && write_floats(f, w) && write_floats(f, m) &&
              write_floats(f, v);
    ok = (std::fclose(f) == 0) && ok;
    return ok ? GLT_OK : io_fail("write failed", path);
}

int glt_nn_load(glt_nn* n, const char* path)
{
    if (!n || !path) return invalid_arg_msg("NULL argument");
    FILE* f = std::fopen(path, "rb");
    if (!f) return io_fail("cannot open", path);
    unsigned char head[8];
    std::vector<float> w, m, v;
    int step = 0;
    int rc = GLT_OK;
    if (std::fread(head, 1, 8, f) != 8) {
        rc = io_fail("short file", path);
    } else if (std::memcmp(head, kCkptTag, 8) == 0) {
        unsigned char b[8];
        if (std::fread(b, 1, 8, f) != 8) {
            rc = io_fail("short checkpoint header", path);
        } else if (le32(b) != kParams || le32(b + 4) < 0) {
            rc = invalid_arg_msg("checkpoint of another network size");
        } else {
            step = le32(b + 4);
            if (!read_floats(f, w, kParams) || !read_floats(f, m, kParams) || !read_floats(f, v, kParams))
                rc = io_fail("short checkpoint", path);
        }
    } else if (std::memcmp(head, "\x93NUMPY", 6) == 0) {
        rc = npy_header(f, head, path);
        if (rc == GLT_OK && !read_floats(f, w, kParams)) rc = io_fail("short .npy data", path);
    } else {
        rc = invalid_arg_msg("neither a network checkpoint nor a .npy file");
    }
    std::fclose(f);
    if (rc != GLT_OK) return rc;
    if (m.empty()) {
        m.assign(kParams, 0.0f);
        v.assign(kParams, 0.0f);
    }
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(n->w, w.data(), kParams * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(n->m, m.data(), kParams * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(n->v, v.data(), kParams * sizeof(float), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "glt_nn_load");
    to_bf16<<<grid_for(kParams, 256), 256>>>(n->w, n->wbf, n->wt);
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_fail(e, "glt_nn_load");
    n->step = step;
    return GLT_OK;
}

}  // extern "C"
