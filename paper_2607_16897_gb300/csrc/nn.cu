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

__device__ __forceinline__ float2 bf2(unsigned v) { return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v)); }

// ---------------------------------------------------------------------------
// Forward pass, convolutions: one persistent block per SM runs conv1-conv3 of
// S samples at a time with all activations and the BF16 weights in shared
// memory, so a sample costs its 4.8 KB of input and 5 KB of features in HBM.
// Bound by FP32 issue: conv2 and conv3 are 5-pixel x CH-channel register tiles
// (per tap and input channel 5 + 1 shared loads for 5 CH FMAs; the lanes of a
// warp share their weights), conv1 8 channels of one pixel.  S = 4 fills the
// shared memory and has the larger tiles; S = 2 has twice the blocks, and is
// taken while those still fit one round (kFwdSmall).  Per output the sum runs
// over the input channels and taps in order, from the bias.  Training also
// stores the activations (a1, a2) that the backward pass reads.  5000 samples:
// 2.03 ms by one thread per output on global memory, 0.27 ms here; 256: 139 ->
// 24 us (caches flushed).
// ---------------------------------------------------------------------------
constexpr int kFwdThreads = 256;
constexpr int kXs = 32 * 42 + 16, kA1s = 16 * 17 * 22 + 16, kA2s = 32 * 10 * 12 + 4;   // per sample: banks staggered
constexpr int kFwdSmall = 2;        // samples per block of the small form

template <int S>
struct FwdSmem {
    float x[S * kXs], a1[S * kA1s], a2[S * kA2s];
    float w1[9 * 16], b1[16], b2[32], b3[64];
    __nv_bfloat16 w2[kW2], w3[kW3];
};

// stride-2 3x3 conv + bias + ReLU of S samples from bordered, column-split
// planes: thread t computes pixels pg + u PG (u < 5) x CH channels of sample s
template <int S, int C, int W, int HO, int WO, int O, int CH, int IN, class Out>
__device__ __forceinline__ void conv_tiles(const float* __restrict__ in, const __nv_bfloat16* __restrict__ w,
                                           const float* __restrict__ bias, Out out)
{
    constexpr int Wp = W + 2, plane = (2 * HO + (W == 20 ? 1 : 2)) * Wp, half = Wp / 2;
    constexpr int PT = 5, PG = HO * WO / PT;
    static_assert(S * PG * (O / CH) == kFwdThreads, "one tile per thread");
    const int t = threadIdx.x;
    const int pg = t % PG, s = (t / PG) % S, cg = t / (PG * S);
    int base[PT];
#pragma unroll
    for (int u = 0; u < PT; ++u) {
        const int p = pg + u * PG;
        base[u] = s * IN + 2 * (p / WO) * Wp + (p % WO);     // window row 2i, split column of 2j
    }
    float acc[PT][CH];
#pragma unroll
    for (int k = 0; k < CH; ++k) {
        const float b = bias[cg * CH + k];
#pragma unroll
        for (int u = 0; u < PT; ++u) acc[u][k] = b;
    }
#pragma unroll 1
    for (int c = 0; c < C; ++c) {
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const __nv_bfloat16* wq = w + (c * 9 + q) * O + cg * CH;
            float wf[CH];
            if (CH == 8) {
                const uint4 r = *reinterpret_cast<const uint4*>(wq);
                const float2 a = bf2(r.x), b = bf2(r.y), d = bf2(r.z), e = bf2(r.w);
                wf[0] = a.x, wf[1] = a.y, wf[2 % CH] = b.x, wf[3 % CH] = b.y;
                wf[4 % CH] = d.x, wf[5 % CH] = d.y, wf[6 % CH] = e.x, wf[7 % CH] = e.y;
            } else if (CH == 4) {
                const uint2 r = *reinterpret_cast<const uint2*>(wq);
                const float2 a = bf2(r.x), b = bf2(r.y);
                wf[0] = a.x, wf[1] = a.y, wf[2 % CH] = b.x, wf[3 % CH] = b.y;
            } else {
                const float2 a = bf2(*reinterpret_cast<const unsigned*>(wq));
                wf[0] = a.x, wf[1] = a.y;
            }
            const int off = c * plane + (q / 3) * Wp + ((q % 3) & 1) * half + ((q % 3) >> 1);   // column 2j + dj
#pragma unroll
            for (int u = 0; u < PT; ++u) {
                const float a = in[base[u] + off];
#pragma unroll
                for (int k = 0; k < CH; ++k) acc[u][k] = fmaf(wf[k], a, acc[u][k]);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < PT; ++u)
#pragma unroll
        for (int k = 0; k < CH; ++k) out(s, cg * CH + k, pg + u * PG, fmaxf(acc[u][k], 0.0f));
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
    for (int b0 = blockIdx.x * S; b0 < B; b0 += gridDim.x * S) {
        for (int i = tid; i < S * kIn; i += kFwdThreads) {
            const int s = i / kIn, p = i - s * kIn, r = p / 40, c = p - r * 40;
            M.x[s * kXs + (r + 1) * 42 + split_col(c + 1, 42)] = b0 + s < B ? x[(size_t)(b0 + s) * kIn + p] : 0.0f;
        }
        __syncthreads();
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
        conv_tiles<S, 16, 20, 8, 10, 32, 2 * S, kA1s>(M.a1, M.w2, M.b2, [&](int s, int o, int p, float r) {
            M.a2[s * kA2s + o * 120 + (p / 10 + 1) * 12 + split_col(p % 10 + 1, 12)] = r;
            if (TRAIN && b0 + s < B) a2g[((size_t)(b0 + s) * 32 + o) * 80 + p] = r;
        });
        __syncthreads();
        conv_tiles<S, 32, 10, 4, 5, 64, S, kA2s>(M.a2, M.w3, M.b3, [&](int s, int o, int p, float r) {
            if (b0 + s < B) a3g[(size_t)(b0 + s) * kFlat + o * 20 + p] = r;
        });
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Fully connected layers of kFcS samples per block: fc1 as 2 outputs x kFcS
// samples per thread, the 1286 inputs split over 8 thread groups (their sums
// added in group order), weights read coalesced from the transposed copy and
// features broadcast from shared memory; then fc2.  In training also the loss
// terms, dy = (y - t) / B, and fc2's input gradient dh (with fc1's ReLU mask).
// Bound by the latency of the weights: 5000 samples 0.67 -> 0.11 ms, 256 52 ->
// 45 us (caches flushed).
// ---------------------------------------------------------------------------
constexpr int kFcS = 8, kFcThreads = 512, kFcSplit = 8;

template <bool TRAIN>
__global__ void __launch_bounds__(kFcThreads)
fc_forward(const float* __restrict__ a3, const float* __restrict__ mo, const __nv_bfloat16* __restrict__ w,
           const __nv_bfloat16* __restrict__ wt, int B, float* __restrict__ y, const float* __restrict__ t,
           float* __restrict__ h, float* __restrict__ dy, float* __restrict__ dh, float* __restrict__ loss_b)
{
    extern __shared__ __align__(16) float smf[];
    float* f = smf;                              // [kFcS][kF + 2]
    float* part = f + kFcS * (kF + 2);           // [kFcSplit][kFcS][kHid]
    __shared__ float hs[kFcS][kHid], ys[kFcS][kOut];
    const int tid = threadIdx.x, b0 = blockIdx.x * kFcS, nb = min(kFcS, B - b0);
    for (int i = tid; i < kFcS * (kF + 2); i += kFcThreads) {
        const int s = i / (kF + 2), k = i - s * (kF + 2);
        float v = 0.0f;
        if (s < nb && k < kF)
            v = k < kFlat ? a3[(size_t)(b0 + s) * kFlat + k] : mo[(size_t)(b0 + s) * kMotion + (k - kFlat)];
        f[i] = v;
    }
    __syncthreads();
    {
        const int o2 = tid & 63, ks = tid >> 6;
        float acc[kFcS][2];
#pragma unroll
        for (int s = 0; s < kFcS; ++s) acc[s][0] = acc[s][1] = 0.0f;
        const __nv_bfloat16* wo = wt + kT4 + 2 * o2;
#pragma unroll 4
        for (int k = 2 * ks; k < kF; k += 2 * kFcSplit) {
            const float2 w0 = bf2(*reinterpret_cast<const unsigned*>(wo + k * kHid));
            const float2 w1 = bf2(*reinterpret_cast<const unsigned*>(wo + (k + 1) * kHid));
#pragma unroll
            for (int s = 0; s < kFcS; ++s) {
                const float2 v = *reinterpret_cast<const float2*>(&f[s * (kF + 2) + k]);
                acc[s][0] = fmaf(w1.x, v.y, fmaf(w0.x, v.x, acc[s][0]));
                acc[s][1] = fmaf(w1.y, v.y, fmaf(w0.y, v.x, acc[s][1]));
            }
        }
#pragma unroll
        for (int s = 0; s < kFcS; ++s)
            *reinterpret_cast<float2*>(&part[(ks * kFcS + s) * kHid + 2 * o2]) = make_float2(acc[s][0], acc[s][1]);
    }
    __syncthreads();
    for (int i = tid; i < kFcS * kHid; i += kFcThreads) {
        float v = 0.0f;
#pragma unroll
        for (int ks = 0; ks < kFcSplit; ++ks) v += part[ks * kFcS * kHid + i];
        v = fmaxf(v + wv(w, kF1.b + i % kHid), 0.0f);
        hs[i / kHid][i % kHid] = v;
        if (TRAIN && i / kHid < nb) h[(size_t)b0 * kHid + i] = v;
    }
    __syncthreads();
    // fc2: warp w computes outputs 4 w .. 4 w + 3 of the 64 (sample, output) pairs
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int q = 0; q < kFcS * kOut / (kFcThreads / 32); ++q) {
        const int e = warp * (kFcS * kOut / (kFcThreads / 32)) + q, s = e / kOut, o = e % kOut;
        float v = 0.0f;
#pragma unroll
        for (int i = 0; i < kHid / 32; ++i) v = fmaf(wv(w, kF2.w + o * kHid + lane + 32 * i), hs[s][lane + 32 * i], v);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        v += wv(w, kF2.b + o);
        if (lane == 0) {
            if (!TRAIN) {
                if (s < nb) y[(size_t)(b0 + s) * kOut + o] = v;
            } else {
                ys[s][o] = s < nb ? v - t[(size_t)(b0 + s) * kOut + o] : 0.0f;
            }
        }
    }
    if (!TRAIN) return;
    __syncthreads();
    if (tid < nb) {
        float e = 0.0f;
#pragma unroll
        for (int o = 0; o < kOut; ++o) e = fmaf(ys[tid][o], ys[tid][o], e);
        loss_b[b0 + tid] = e;
    }
    if (tid < nb * kOut) dy[(size_t)b0 * kOut + tid] = ys[tid / kOut][tid % kOut] / (float)B;
    for (int i = tid; i < nb * kHid; i += kFcThreads) {
        const int s = i / kHid, k = i % kHid;
        float v = 0.0f;
#pragma unroll
        for (int o = 0; o < kOut; ++o) v = fmaf(wv(w, kF2.w + o * kHid + k), ys[s][o] / (float)B, v);
        dh[(size_t)b0 * kHid + i] = hs[s][k] > 0.0f ? v : 0.0f;
    }
}

// d3[b,i] = (sum_o fc1.w[o,i] dh[b,o]) (a3[b,i] > 0) for the 1280 conv3
// features: 8 samples x 2 features per thread, 256 features per block.
constexpr int kD3Threads = 128;

__global__ void __launch_bounds__(kD3Threads)
fc1_input_grad(const float* __restrict__ dh, const __nv_bfloat16* __restrict__ w, const float* __restrict__ a3, int B,
               float* __restrict__ d3)
{
    __shared__ __align__(16) float d[kFcS][kHid];
    const int tid = threadIdx.x, b0 = blockIdx.x * kFcS, nb = min(kFcS, B - b0);
    for (int i = tid; i < kFcS * kHid; i += kD3Threads) d[i / kHid][i % kHid] = i / kHid < nb ? dh[(size_t)b0 * kHid + i] : 0.0f;
    __syncthreads();
    const int i = 2 * (blockIdx.y * kD3Threads + tid);
    float acc[kFcS][2];
#pragma unroll
    for (int s = 0; s < kFcS; ++s) acc[s][0] = acc[s][1] = 0.0f;
#pragma unroll 2
    for (int o = 0; o < kHid; o += 4) {
        float2 wf[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) wf[q] = bf2(*reinterpret_cast<const unsigned*>(w + kF1.w + (o + q) * kF + i));
#pragma unroll
        for (int s = 0; s < kFcS; ++s) {
            const float4 v = *reinterpret_cast<const float4*>(&d[s][o]);
            const float vq[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                acc[s][0] = fmaf(wf[q].x, vq[q], acc[s][0]);
                acc[s][1] = fmaf(wf[q].y, vq[q], acc[s][1]);
            }
        }
    }
#pragma unroll
    for (int s = 0; s < kFcS; ++s) {
        if (s >= nb) break;
        const size_t at = (size_t)(b0 + s) * kFlat + i;
        const float2 a = *reinterpret_cast<const float2*>(a3 + at);
        *reinterpret_cast<float2*>(d3 + at) = make_float2(a.x > 0.0f ? acc[s][0] : 0.0f, a.y > 0.0f ? acc[s][1] : 0.0f);
    }
}

// Weight and bias gradients of the fully connected layers: dW[o,i] = sum_b
// dz[b,o] in[b,i], the bias as one more input of ones.  32 x 32 output tiles,
// 4 x 4 per thread, 32 samples staged at a time; the tiles of fc1 (4 x 41)
// come first, then fc2's (1 x 5).
constexpr int kGwThreads = 64, kGwT = 32;
constexpr int kGwI1 = (kF + 1 + kGwT - 1) / kGwT, kGwI2 = (kHid + 1 + kGwT - 1) / kGwT;
constexpr int kGwBlocks = (kHid / kGwT) * kGwI1 + kGwI2;

__global__ void __launch_bounds__(kGwThreads)
fc_weight_grad(const float* __restrict__ dh, const float* __restrict__ dy, const float* __restrict__ a3,
               const float* __restrict__ mo, const float* __restrict__ h, int B, float* __restrict__ grad)
{
    __shared__ __align__(16) float zs[kGwT][kGwT], is[kGwT][kGwT];
    const bool first = blockIdx.x < (kHid / kGwT) * kGwI1;
    const int tile = first ? blockIdx.x : blockIdx.x - (kHid / kGwT) * kGwI1;
    const int O = first ? kHid : kOut, n = first ? kF : kHid;
    const int o0 = first ? (tile / kGwI1) * kGwT : 0, i0 = (first ? tile % kGwI1 : tile) * kGwT;
    const float* dz = first ? dh : dy;
    const int tid = threadIdx.x, to = (tid / 8) * 4, ti = (tid % 8) * 4;
    float acc[4][4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = 0.0f;
    for (int b0 = 0; b0 < B; b0 += kGwT) {
#pragma unroll 8
        for (int e = tid; e < kGwT * kGwT; e += kGwThreads) {
            const int b = b0 + e / kGwT, o = o0 + e % kGwT, i = i0 + e % kGwT;
            float z = 0.0f, v = 0.0f;
            if (b < B) {
                if (o < O) z = dz[(size_t)b * O + o];
                if (i == n)
                    v = 1.0f;
                else if (i < n)
                    v = !first ? h[(size_t)b * kHid + i] : i < kFlat ? a3[(size_t)b * kFlat + i]
                                                                   : mo[(size_t)b * kMotion + (i - kFlat)];
            }
            zs[e / kGwT][e % kGwT] = z;
            is[e / kGwT][e % kGwT] = v;
        }
        __syncthreads();
#pragma unroll 8
        for (int b = 0; b < kGwT; ++b) {
            const float4 z = *reinterpret_cast<const float4*>(&zs[b][to]);
            const float4 v = *reinterpret_cast<const float4*>(&is[b][ti]);
            const float zq[4] = {z.x, z.y, z.z, z.w}, vq[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(zq[p], vq[q], acc[p][q]);
        }
        __syncthreads();
    }
    const int woff = first ? kF1.w : kF2.w, boff = first ? kF1.b : kF2.b;
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int o = o0 + to + p, i = i0 + ti + q;
            if (o >= O || i > n) continue;
            grad[i == n ? boff + o : woff + o * n + i] = acc[p][q];
        }
}

// ---------------------------------------------------------------------------
// Backward pass of the convolutions: a block takes whole samples, one at a
// time, keeps their activations and gradients in shared memory, and carries
// its weight-gradient sums in registers over all of them; the blocks' sums go
// to `part` and are added in block order by adam_update.  Bound by FP32 issue
// and the shared-memory pipe.
//  * input gradients (d2 from d3, d1 from d2): a thread owns a 2 x 2 quad of
//    input pixels x 4 channels, whose nine (pixel, tap) pairs use each weight
//    once (36 FMAs per 9 + 4 shared loads); conv3's 64 channels are split over
//    two thread groups;
//  * weight gradients: a thread owns 8 output channels x the 9 taps of one
//    input channel (72 sums; 72 FMAs per 2 + 9 shared loads): half of the
//    block conv3's, the other half conv2's with the positions split over four
//    thread groups; conv1 one (channel, row) per thread.
// Input planes have an odd stride, so the lanes of a warp (channels) read
// different banks.  256 samples: 82 us, against 1.43 ms of one block per weight
// and one thread per input value on global memory.
// ---------------------------------------------------------------------------
constexpr int kBwThreads = 512, kBwBlocks = 148;
constexpr int kP1 = 375, kP2 = 121;                       // plane strides of a1 (17 x 22) and a2 (10 x 12)
constexpr int kPart = kW3 + 64 + kW2 + 32 + 144 + 16;     // one block's sums: conv3, conv2, conv1 (w, b each)
constexpr int kPt3 = 0, kPt2 = kW3 + 64, kPt1 = kPt2 + kW2 + 32;

struct BwdSmem {
    float w3[kW3], w2[kW2];             // [output channel][tap][input channel]
    float x[32 * 42], a1[16 * kP1], a2[32 * kP2];
    float d3[20 * 64];                  // [position][channel]
    float d3p[64 * 30];                 // [channel][5 x 6], zero beyond 4 x 5
    float d2[80 * 32];                  // [position][channel]
    float d2p[32 * 99];                 // [channel][9 x 11], zero beyond 8 x 10
    float d1[16 * 301];                 // [channel][15 x 20]
    float tmp[160 * 16];                // the second half of conv3's input gradient
};

// the quad (i0, j0) of an input gradient: acc[px][channel] over output
// channels [o0, o1); dp: padded gradient planes of stride DP and row DW;
// w: [o][tap][C]
template <int C, int DP, int DW>
__device__ __forceinline__ void quad_grad(const float* __restrict__ dp, const float* __restrict__ w, int o0, int o1,
                                          int i0, int j0, int c0, float (&acc)[4][4])
{
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[p][k] = 0.0f;
#pragma unroll 2
    for (int o = o0; o < o1; ++o) {
        const float* d = dp + o * DP + i0 * DW + j0;
        const float d00 = d[0], d01 = d[1], d10 = d[DW], d11 = d[DW + 1];
        const float* wo = w + o * 9 * C + c0;
        // input row 2 i0 takes tap row 1 of output row i0; row 2 i0 + 1 tap row
        // 2 of i0 and tap row 0 of i0 + 1; columns alike
        auto tap = [&](int q, int px, float v) {
            const float4 r = *reinterpret_cast<const float4*>(wo + q * C);
            acc[px][0] = fmaf(r.x, v, acc[px][0]);
            acc[px][1] = fmaf(r.y, v, acc[px][1]);
            acc[px][2] = fmaf(r.z, v, acc[px][2]);
            acc[px][3] = fmaf(r.w, v, acc[px][3]);
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
}

// weight-gradient sums of 8 output channels x 9 taps of one input plane over
// positions [p0, p1)
template <int WO, int Wp, int O>
__device__ __forceinline__ void tap_grad(const float* __restrict__ dpos, const float* __restrict__ plane, int p0, int p1,
                                         int og, float (&acc)[8][9], float (&bias)[8])
{
    for (int p = p0; p < p1; ++p) {
        const float4 da = *reinterpret_cast<const float4*>(dpos + p * O + og * 8);
        const float4 db = *reinterpret_cast<const float4*>(dpos + p * O + og * 8 + 4);
        const float dv[8] = {da.x, da.y, da.z, da.w, db.x, db.y, db.z, db.w};
        const float* in = plane + 2 * (p / WO) * Wp + (p % WO);
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float v = in[(q / 3) * Wp + ((q % 3) & 1) * (Wp / 2) + ((q % 3) >> 1)];
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k][q] = fmaf(dv[k], v, acc[k][q]);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) bias[k] += dv[k];
    }
}

__global__ void __launch_bounds__(kBwThreads, 1)
conv_backward(const float* __restrict__ x, const float* __restrict__ a1, const float* __restrict__ a2,
              const float* __restrict__ d3, const __nv_bfloat16* __restrict__ wt, int B, float* __restrict__ part)
{
    extern __shared__ __align__(16) unsigned char raw[];
    BwdSmem& M = *reinterpret_cast<BwdSmem*>(raw);
    const int tid = threadIdx.x;
    for (int i = tid; i < kW3; i += kBwThreads) M.w3[i] = wv(wt, kB3 + i);
    for (int i = tid; i < kW2; i += kBwThreads) M.w2[i] = wv(wt, kB2 + i);
    for (int i = tid; i < (int)((sizeof(BwdSmem) - offsetof(BwdSmem, x)) / sizeof(float)); i += kBwThreads) M.x[i] = 0.0f;
    // weight-gradient roles: threads 0-255 conv3 (8 output groups x 32 input
    // channels), the others conv2 (4 position groups x 4 x 16)
    const bool third = tid < 256;
    const int u = tid & 255, gc = third ? u & 31 : u & 15, gg = third ? u >> 5 : (u >> 4) & 3, gs = u >> 6;
    const int o1 = tid & 15, r1 = tid >> 4;               // conv1: channel, row (r1 < 15)
    float wg[8][9], bg[8], w1g[9], b1g = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        bg[k] = 0.0f;
#pragma unroll
        for (int q = 0; q < 9; ++q) wg[k][q] = 0.0f;
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) w1g[q] = 0.0f;
    __syncthreads();
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        for (int i = tid; i < kIn; i += kBwThreads) M.x[(i / 40 + 1) * 42 + split_col(i % 40 + 1, 42)] = x[(size_t)b * kIn + i];
        for (int i = tid; i < 4800; i += kBwThreads) {
            const int c = i / 300, p = i % 300;
            M.a1[c * kP1 + (p / 20 + 1) * 22 + split_col(p % 20 + 1, 22)] = a1[(size_t)b * 4800 + i];
        }
        for (int i = tid; i < 2560; i += kBwThreads) {
            const int c = i / 80, p = i % 80;
            M.a2[c * kP2 + (p / 10 + 1) * 12 + split_col(p % 10 + 1, 12)] = a2[(size_t)b * 2560 + i];
        }
        for (int i = tid; i < kFlat; i += kBwThreads) {
            const int o = i / 20, p = i % 20;
            const float v = d3[(size_t)b * kFlat + i];
            M.d3[p * 64 + o] = v;
            M.d3p[o * 30 + (p / 5) * 6 + p % 5] = v;
        }
        __syncthreads();
        // d2, in two halves of conv3's channels
        {
            const int half = tid / 160, e = tid % 160, quad = e % 20, cg = e / 20;
            const int i0 = quad / 5, j0 = quad % 5;
            float acc[4][4];
            if (half < 2) quad_grad<32, 30, 6>(M.d3p, M.w3, half * 32, half * 32 + 32, i0, j0, cg * 4, acc);
            if (half == 1) {
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int k = 0; k < 4; ++k) M.tmp[(p * 4 + k) * 160 + e] = acc[p][k];
            }
            __syncthreads();
            if (half == 0) {
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const int yy = 2 * i0 + (p >> 1), xx = 2 * j0 + (p & 1);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int c = cg * 4 + k;
                        const bool on = M.a2[c * kP2 + (yy + 1) * 12 + split_col(xx + 1, 12)] > 0.0f;
                        const float v = on ? acc[p][k] + M.tmp[(p * 4 + k) * 160 + e] : 0.0f;
                        M.d2[(yy * 10 + xx) * 32 + c] = v;
                        M.d2p[c * 99 + yy * 11 + xx] = v;
                    }
                }
            }
        }
        __syncthreads();
        if (third)
            tap_grad<5, 12, 64>(M.d3, M.a2 + gc * kP2, 0, 20, gg, wg, bg);
        else
            tap_grad<10, 22, 32>(M.d2, M.a1 + gc * kP1, gs * 20, gs * 20 + 20, gg, wg, bg);
        if (tid < 320) {
            const int quad = tid % 80, cg = tid / 80, i0 = quad / 10, j0 = quad % 10;
            float acc[4][4];
            quad_grad<16, 99, 11>(M.d2p, M.w2, 0, 32, i0, j0, cg * 4, acc);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int yy = 2 * i0 + (p >> 1), xx = 2 * j0 + (p & 1);
                if (yy >= 15) continue;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int c = cg * 4 + k;
                    const bool on = M.a1[c * kP1 + (yy + 1) * 22 + split_col(xx + 1, 22)] > 0.0f;
                    M.d1[c * 301 + yy * 20 + xx] = on ? acc[p][k] : 0.0f;
                }
            }
        }
        __syncthreads();
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
    float* red = M.w3;                                   // 4 x (kW2 + 32), then 15 x 160
    if (third) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
#pragma unroll
            for (int q = 0; q < 9; ++q) out[kPt3 + ((gg * 8 + k) * 32 + gc) * 9 + q] = wg[k][q];
            if (gc == 0) out[kPt3 + kW3 + gg * 8 + k] = bg[k];
        }
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
#pragma unroll
            for (int q = 0; q < 9; ++q) red[gs * kW2 + ((gg * 8 + k) * 16 + gc) * 9 + q] = wg[k][q];
            if (gc == 0) M.tmp[gs * 32 + gg * 8 + k] = bg[k];
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
// block order over four interleaved quarters) and, with ADAM, the update
// (Kingma and Ba) of the FP32 master weights and the BF16 copies.  Blocks
// below kAdConv take 64 convolution parameters each, four threads per
// parameter; the rest 256 parameters of the fully connected layers; the last
// one adds the loss terms.
constexpr int kAdConvN = kPart, kAdConv = (kAdConvN + 63) / 64;
constexpr int kAdFc = (kParams - kF1.w + 255) / 256, kAdBlocks = kAdConv + kAdFc + 1;
static_assert(kAdConvN == kF1.w, "the convolutions' parameters come first");

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
        __shared__ float q4[4][64];
        const int e = threadIdx.x & 63, q = threadIdx.x >> 6, c = blockIdx.x * 64 + e;
        // parameter c in file order (conv1.w, conv1.b, conv2.w, ...) -> its place in a block's sums
        const int at = c < 160 ? kPt1 + c : c < kC3.w ? kPt2 + c - kC2.w : kPt3 + c - kC3.w;
        float s = 0.0f;
        if (c < kAdConvN) {
#pragma unroll 8
            for (int k = q; k < nparts; k += 4) s += part[(size_t)k * kPart + at];
        }
        q4[q][e] = s;
        __syncthreads();
        if (q == 0 && c < kAdConvN) {
            i = c;
            gi = ((q4[0][e] + q4[1][e]) + q4[2][e]) + q4[3][e];
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
          *d3 = nullptr, *part = nullptr, *loss_b = nullptr;
    float* loss = nullptr;
};

using namespace glt;
using namespace glt::nn;

namespace {

constexpr size_t kFcSmem = (size_t)(kFcS * (kF + 2) + kFcSplit * kFcS * kHid) * sizeof(float);

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
    if (e == cudaSuccess) e = al(&n->part, (size_t)std::min(B, kBwBlocks) * kPart);
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
    if (e == cudaSuccess) e = smem(fc_forward<false>, kFcSmem);
    if (e == cudaSuccess) e = smem(fc_forward<true>, kFcSmem);
    if (e == cudaSuccess) e = smem(conv_backward, sizeof(BwdSmem));
    return e == cudaSuccess ? GLT_OK : cuda_fail(e, "proposal network allocation");
}

void nn_free(glt_nn* n)
{
    if (!n) return;
    for (float* p : {n->w, n->g, n->m, n->v, n->a1, n->a2, n->a3, n->h, n->y, n->dy, n->dh, n->d3, n->part, n->loss_b,
                     n->loss})
        cudaFree(p);
    cudaFree(n->wbf);
    cudaFree(n->wt);
    delete n;
}

int grid_for(int n, int t) { return (n + t - 1) / t; }

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

cudaError_t nn_forward(const glt_nn* n, const float* x, const float* mo, int B, float* y, cudaStream_t s)
{
    launch_conv_forward<false>(n, x, B, s);
    fc_forward<false><<<grid_for(B, kFcS), kFcThreads, kFcSmem, s>>>(n->a3, mo, n->wbf, n->wt, B, y, nullptr, nullptr,
                                                                     nullptr, nullptr, nullptr);
    return cudaGetLastError();
}

// forward and backward: the gradient sums up to adam_update, which completes them
cudaError_t nn_backward(const glt_nn* n, const float* x, const float* mo, const float* t, int B, cudaStream_t s)
{
    launch_conv_forward<true>(n, x, B, s);
    fc_forward<true><<<grid_for(B, kFcS), kFcThreads, kFcSmem, s>>>(n->a3, mo, n->wbf, n->wt, B, n->y, t, n->h, n->dy,
                                                                    n->dh, n->loss_b);
    fc1_input_grad<<<dim3(grid_for(B, kFcS), kFlat / (2 * kD3Threads)), kD3Threads, 0, s>>>(n->dh, n->wbf, n->a3, B, n->d3);
    fc_weight_grad<<<kGwBlocks, kGwThreads, 0, s>>>(n->dh, n->dy, n->a3, mo, n->h, B, n->g);
    conv_backward<<<std::min(B, kBwBlocks), kBwThreads, sizeof(BwdSmem), s>>>(x, n->a1, n->a2, n->d3, n->wt, B, n->part);
    return cudaGetLastError();
}

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
// the start and awaited just before conv2.  The sum order per output (bias,
// then channel, row, column) is that of conv_fwd.
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
// per stream.  Each output keeps conv_fwd's lane split and reduction order.
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
    // an output that overlaps an input is written when all inputs have been read
    auto overlap = [&](const float* p, size_t len) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(p), b = reinterpret_cast<uintptr_t>(y_dev);
        return a < b + (size_t)B * kOut * sizeof(float) && b < a + len * sizeof(float);
    };
    const bool staged = overlap(x_dev, (size_t)B * kIn) || overlap(m_dev, (size_t)B * kMotion);
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
        adam_update<false><<<kAdBlocks, 256, 0, s>>>(n->w, n->wbf, n->wt, n->g, n->part, std::min(B, kBwBlocks), n->m, n->v,
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
    const double b1 = 0.9, b2 = 0.999;
    const float c1 = (float)(1.0 / (1.0 - std::pow(b1, n->step)));
    const float c2 = (float)(1.0 / (1.0 - std::pow(b2, n->step)));
    adam_update<true><<<kAdBlocks, 256, 0, s>>>(n->w, n->wbf, n->wt, n->g, n->part, std::min(B, kBwBlocks), n->m, n->v, lr,
                                                (float)b1, (float)b2, 1e-8f, c1, c2, n->loss_b, B,
                                                loss_dev ? loss_dev : n->loss);
    if (e == cudaSuccess) e = cudaGetLastError();
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
