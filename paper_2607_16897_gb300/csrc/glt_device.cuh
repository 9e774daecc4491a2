// Device-side building blocks of the tracker: per-stream descriptors, the
// per-point linearisation (projection, bilinear gather of I and grad I,
// residual, Huber weight, forward Jacobian, 44-term normal-equation
// accumulation), the warp reduce-scatter, and the FP64 LM solver tail
// (Cholesky 8x8, SE(3) exponential, pose composition).
//
// Method: GLidE-SLAM Sec. IV (Eqs. 1-5) in the forward form of Sec. IV-B
// (Jacobian from the current image's gradient at the warped location), with
// affine brightness, Huber weights and LM damping added by this library.
#pragma once

#include <type_traits>
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>

#include "glt.h"

namespace glt {

constexpr int kMaxLevels = GLT_MAX_LEVELS;
constexpr int kNumH = 36;        // upper triangle of the 8x8 H
constexpr int kIdxG = 36;        // g = J^T W r, 8 entries
constexpr int kIdxE = 44;        // Huber energy
constexpr int kIdxN = 45;        // valid sample count
constexpr int kNumAcc = 46;
constexpr int kAccPad = 48;      // padded for the 5-stage reduce-scatter
// cached-Hessian form: g0 = sum w r J_ic (6), Huber energy, sample count
constexpr int kHcAcc = 8;
constexpr int kHcE = 6;
constexpr int kHcN = 7;

// 8-pixel sparse pattern (offsets du_k of Eq. 2), level pixels.
__host__ __device__ constexpr int pat_dx(int k) { return k == 1 ? -2 : k == 2 ? 2 : k == 5 ? -1 : k == 6 ? 1 : k == 7 ? -1 : 0; }
__host__ __device__ constexpr int pat_dy(int k) { return k == 3 ? -2 : k == 4 ? 2 : (k == 5 || k == 6) ? -1 : k == 7 ? 1 : 0; }

// Programmatic dependent launch (sm_90 and later): a kernel launched with
// cudaLaunchAttributeProgrammaticStreamSerialization may begin while the
// previous kernel of its stream still runs.  griddep_wait() returns once that
// kernel has completed and its writes are visible; griddep_launch_dependents()
// lets the next such kernel begin.  Both are no-ops for an ordinary launch.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The uint8 CUR levels may be written by a pyramid kernel that was still
// running when the track kernel started (a programmatic dependent launch), so
// the gathers read them with ld.global.ca (weak, L1-cached loads ordered by
// the dependency wait), never through the read-only path, which assumes data
// that is final for the whole lifetime of the kernel.
struct LevelDev {
    const uint8_t* img;   // uint8 level, `pitch` bytes per row (pitch >= W + 8, multiple of 16)
    const uint2* packed;  // GLT_MIXED: FP16 (I, gx, gy, 0) per pixel, W pixels per row
    int W, H, pitch;
};

// One tracked stream as the kernels see it (device memory).
struct StreamDesc {
    LevelDev lv[kMaxLevels];
    int L, N, Npad;
    float fx, fy;          // level-0 focal lengths
    float huber_k, zmin;
    const float4* pt;      // (u0, v0, (u0-cx)/fx, (v0-cy)/fy)
    const float2* dz;      // (depth, 1/depth)
    const float* I0;       // reference samples, in the order of table_index; a point's first
                           // sample is NaN on a level where it is unusable
    const float2* G0;      // GLT_IC: reference gradients (gx, gy) in the same order, else null
    int pattern, K;        // 0 and 8: the 8-pixel pattern; p and p*p: the p x p patch
    int tg;                // p x p patches: threads that share a point (hc_groups, else 1)
    int affine;            // 0: (a, b) held at their initial values
    const double* Hc;      // GLT_HESSIAN_CACHED: per level H (36) then H^-1 (36), row-major
                           // 6x6 pose blocks of the reference rows; H^-1[0] NaN if H is not PD
    int max_iters[kMaxLevels];
    int min_valid;
    int max_trace;
    double lambda0, lambda_up, lambda_down, eps_step, eps_step_coarse, eps_cost, accept_step;
    double* trace_E;       // [max_trace] Huber energy of each pass, or null
    int* trace_n;          // [max_trace] valid samples of each pass
    int* trace_info;       // [max_trace] level * 4 + 2 * accepted + is_candidate
    int* trace_count;      // passes of the last track, or null
    int solve;             // GLT_SOLVE_FP64 or GLT_SOLVE_FP32
};

// The cached-Hessian form splits a 7 x 7 or 11 x 11 patch into kHcGroups
// groups of consecutive rows, one thread per group.
constexpr int kHcGroups = 4;
__host__ __device__ constexpr int hc_groups(int pattern) { return (pattern == 7 || pattern == 11) ? kHcGroups : 1; }
// rows and samples of a group of a p x p patch shared by tg threads
__host__ __device__ constexpr int group_rows(int pattern, int tg) { return (pattern + tg - 1) / tg; }
__host__ __device__ constexpr int group_samples(int pattern, int tg) { return group_rows(pattern, tg) * pattern; }

// Order of the reference tables.  The 8-pixel pattern keeps a point's 8 samples
// together (one 32-byte read per point).  A p x p patch is stored sample by
// sample over the tasks (point, group), so that the lanes of a warp, which work
// on consecutive tasks, read consecutive words: point by point a lane's reads
// lay K words apart and every load cost a wavefront per point.  With the UNIT
// sums of linearize_rows_hc and the L1 kept over the cluster's exchange: 7.0k ->
// 4.1k cycles to linearise 2000 points of a pass at 7 x 7, 13.6k -> 6.3k at
// 11 x 11; with a Huber threshold 66 passes take 438 instead of 554 us at 7 x 7,
// 700 instead of 860 at 11 x 11, 561 and 1390 at 5 x 5 and 9 x 9 instead of 1127
// and 2920 (then per-pixel byte loads).
__host__ __device__ inline size_t table_size(int L, int Npad, int pattern, int tg)
{
    return pattern ? (size_t)L * group_samples(pattern, tg) * Npad * tg : (size_t)L * Npad * 8;
}

// Bounds-checked build (compiled with -DGLT_CHECKED into libglt_checked.so):
// every gather and table access of the hot path checks its element range
// [p, p + n) against its buffer [base, base + size); an access outside sets
// bit `site` of this translation unit's check flags and goes to the buffer's
// first element instead (no trap, no access outside the buffer).  In the
// normal build checked() is the pointer itself.
enum CheckSite {
    CK_IMAGE = 0,      // uint8 level window rows
    CK_PACKED = 1,     // FP16-packed level texels
    CK_TABLE = 2,      // per-point reference tables (I0, G0)
    CK_POINTS = 3,     // point arrays (pt, dz)
    CK_PYR_SRC = 4,    // pyramid source rows
    CK_PYR_DST = 5,    // pyramid destination and level-0 copy
    CK_SET_POINTS = 6  // reference-table writes of set_points
};
#ifdef GLT_CHECKED
static __device__ unsigned g_check_flags;
template <class T>
__device__ __forceinline__ T* checked(T* p, size_t n, T* base, size_t size, int site)
{
    if (p < base || p + n > base + size) {
        atomicOr(&g_check_flags, 1u << site);
        return base;
    }
    return p;
}
#else
template <class T>
__device__ __forceinline__ T* checked(T* p, size_t, T*, size_t, int)
{
    return p;
}
#endif

// The state one linearisation pass is evaluated at, in the form the FP32
// gather uses: R - I and t rounded from the FP64 pose, e^a, b.
struct PassParams {
    float Rm[9];           // the first 14 floats are also written by index (tail_map_init)
    float t[3];
    float ea, b;
    float scale;           // 2^-level
    int level;
    int done;
};

// ---------------------------------------------------------------------------
// Per-point linearisation
// ---------------------------------------------------------------------------
// Byte `byte` of w as a float: 2^23 + byte through the bits (0x4b0000bb), minus
// 2^23 (exact).  3.7 cycles of a sub-partition with the add that uses it, where
// the conversion took 4.3 (and 4.2 against 7.4 with one warp).
__device__ __forceinline__ float u8f(uint32_t w, int byte)
{
    return __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7540 | byte)) - 8388608.0f;
}

struct PointGeom {
    float al, be;          // bilinear weights' fractions (shared by all 8 samples)
    int xb, yb;            // integer base of sample 0
    float a0[3], a1[3];    // rows of d(pi)/d(x_c) * R (level intrinsics)
    float xr[3];           // x_r
};

// Projects point p through the pass state. Returns false if the point is not
// usable (invalid reference, behind zmin, or a pattern sample outside
// 1 <= q < W-2, 1 <= q < H-2).
//
// Projection is evaluated relative to the reference pixel to keep FP32
// accurate at any image width:  with m = ((u0-cx)/fx, (v0-cy)/fy, 1) and
// D = (R - I) m + t / d,  x_c = d (m + D)  and
// u - u0 = fx (D_x - m_x D_z) / (1 + D_z)   (exactly Eq. 1's pi(R x_r + t)).
// A point's data for one level: position, depth, reference patch (I0[0..7];
// for a p x p patch only I0[0], the validity marker).  Loaded once per level
// and kept across that level's passes when a thread owns a single point.
struct PointCache {
    float4 q;
    float2 dz;
    float4 ia, ib;
    int p, level;
};

// Sample (row j, column i) of the p x p patch of point p on a level.
template <int PS, int TG>
__device__ __forceinline__ size_t patch_index(const StreamDesc& D, int level, int p, int j, int i)
{
    constexpr int RG = group_rows(PS, TG), SG = group_samples(PS, TG);
    const int g = j / RG;
    return ((size_t)level * SG + (j - g * RG) * PS + i) * ((size_t)D.Npad * TG) + (size_t)p * TG + g;
}
// ... of a patch of any size that one thread works on (tg = 1)
__device__ __forceinline__ size_t patch_index1(const StreamDesc& D, int level, int p, int k)
{
    return ((size_t)level * D.K + k) * D.Npad + p;
}
// tab + i, from where n elements are read
template <class T>
__device__ __forceinline__ const T* table_from(const StreamDesc& D, const T* tab, size_t i, size_t n)
{
    return checked(tab + i, n, tab, table_size(D.L, D.Npad, D.pattern, D.tg), CK_TABLE);
}

__device__ __forceinline__ void load_point(const StreamDesc& D, int level, int p, PointCache& c)
{
    c.q = *checked(D.pt + p, 1, D.pt, (size_t)D.Npad, CK_POINTS);
    c.dz = *checked(D.dz + p, 1, D.dz, (size_t)D.Npad, CK_POINTS);
    if (D.pattern) {
        // the p x p path reads its samples itself; the first marks validity
        const size_t at = ((size_t)level * group_samples(D.pattern, D.tg) * D.Npad + p) * D.tg;
        c.ia = make_float4(*table_from(D, D.I0, at, 1), 0.f, 0.f, 0.f);
        c.ib = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
        const float* I0b = checked(D.I0 + ((size_t)level * D.Npad + p) * 8, 8, D.I0, (size_t)D.L * D.Npad * 8, CK_TABLE);
        const float4* I0p = reinterpret_cast<const float4*>(I0b);   // K = 8: 32-byte rows
        c.ia = I0p[0];
        c.ib = I0p[1];
    }
    c.p = p;
    c.level = level;
}

template <bool SQUARE = false>
__device__ __forceinline__ bool project_point(const StreamDesc& D, const PassParams& P,
                                              const LevelDev& lv, const PointCache& c, PointGeom& G)
{
    const float4 q = c.q;
    const float2 dz = c.dz;
    const float ub = q.z, vb = q.w, d = dz.x, rho = dz.y;
    const float Dx = fmaf(P.Rm[0], ub, fmaf(P.Rm[1], vb, fmaf(P.t[0], rho, P.Rm[2])));
    const float Dy = fmaf(P.Rm[3], ub, fmaf(P.Rm[4], vb, fmaf(P.t[1], rho, P.Rm[5])));
    const float Dz = fmaf(P.Rm[6], ub, fmaf(P.Rm[7], vb, fmaf(P.t[2], rho, P.Rm[8])));
    const float onez = 1.0f + Dz;
    if (!(d * onez > D.zmin)) return false;
    const float iz = 1.0f / onez;
    const float du = D.fx * fmaf(-ub, Dz, Dx) * iz;
    const float dv = D.fy * fmaf(-vb, Dz, Dy) * iz;
    if (!(fabsf(du) < 1e6f && fabsf(dv) < 1e6f)) return false;
    const float s = P.scale;
    const float U = q.x * s, V = q.y * s;
    const float Ui = floorf(U), Vi = floorf(V);
    const float su = (U - Ui) + du * s;
    const float sv = (V - Vi) + dv * s;
    const float fu = floorf(su), fv = floorf(sv);
    G.al = su - fu;
    G.be = sv - fv;
    G.xb = (int)Ui + (int)fu;
    G.yb = (int)Vi + (int)fv;
    const int h = (SQUARE && D.pattern) ? (D.pattern - 1) / 2 : 2;   // half extent of the pattern
    if (G.xb < 1 + h || G.xb > lv.W - 3 - h || G.yb < 1 + h || G.yb > lv.H - 3 - h) return false;
    // d(pi)/d(x_c) R, with x_c / z_c = (m + D) / (1 + D_z) and 1/z_c = rho / (1 + D_z)
    const float xn = (ub + Dx) * iz, yn = (vb + Dy) * iz;
    const float fxl = D.fx * s * rho * iz, fyl = D.fy * s * rho * iz;
    const float R0[3] = {1.0f + P.Rm[0], P.Rm[1], P.Rm[2]};
    const float R1[3] = {P.Rm[3], 1.0f + P.Rm[4], P.Rm[5]};
    const float R2[3] = {P.Rm[6], P.Rm[7], 1.0f + P.Rm[8]};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        G.a0[c] = fxl * fmaf(-xn, R2[c], R0[c]);
        G.a1[c] = fyl * fmaf(-yn, R2[c], R1[c]);
    }
    G.xr[0] = d * ub;
    G.xr[1] = d * vb;
    G.xr[2] = d;
    return true;
}

// Accumulates one residual sample into acc (upper triangle of w J J^T, w J r,
// Huber energy, count).
// COUNT: also the sample (the 8-pixel pattern counts a point's 8 at once: the
// counts are whole numbers, exact either way).
template <bool COUNT = true>
__device__ __forceinline__ void accumulate_sample(const PointGeom& G, float I, float gx, float gy,
                                                  float i0, float ea, float b, float k,
                                                  float* acc, float* res_out)
{
    float J[8];
    const float Jt0 = fmaf(gx, G.a0[0], gy * G.a1[0]);
    const float Jt1 = fmaf(gx, G.a0[1], gy * G.a1[1]);
    const float Jt2 = fmaf(gx, G.a0[2], gy * G.a1[2]);
    J[0] = Jt0;
    J[1] = Jt1;
    J[2] = Jt2;
    // rotational columns: row vector (Jt) * (-[x_r]x) = x_r x Jt
    J[3] = fmaf(G.xr[1], Jt2, -G.xr[2] * Jt1);
    J[4] = fmaf(G.xr[2], Jt0, -G.xr[0] * Jt2);
    J[5] = fmaf(G.xr[0], Jt1, -G.xr[1] * Jt0);
    J[6] = -ea * i0;
    J[7] = -1.0f;
    const float r = fmaf(-ea, i0, I) - b;
    const float ar = fabsf(r);
    const float w = ar <= k ? 1.0f : k / ar;
    const float rho = ar <= k ? 0.5f * r * r : k * (ar - 0.5f * k);
    if (res_out) *res_out = r;
    float wJ[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) wJ[i] = w * J[i];
    int idx = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
        for (int j = i; j < 8; ++j) {
            acc[idx] = fmaf(wJ[i], J[j], acc[idx]);
            ++idx;
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[kIdxG + i] = fmaf(wJ[i], r, acc[kIdxG + i]);
    acc[kIdxE] += rho;
    if (COUNT) acc[kIdxN] += 1.0f;
}

// Cached-Hessian form (Sec. IV-B: with the rows on the reference side H is
// fixed per reference and level; Sec. IV-C "Track": each point contributes
// only its right-hand side b_i = -sum_k J_ik^T r_ik).  A sample adds its
// Huber-weighted residual times the cached reference gradient to the point's
// (sx, sy); the point then folds them into g0 = sum w r J_ic:
// J_k = [Jt_k, x_r x Jt_k] with Jt_k = gx_k a0 + gy_k a1, so
// sum_k w_k r_k J_k = [v, x_r x v] with v = sx a0 + sy a1.
__device__ __forceinline__ void hc_sample(float I, float i0, float2 g0, float ea, float b, float k,
                                          float& sx, float& sy, float* acc, float* res_out)
{
    const float r = fmaf(-ea, i0, I) - b;
    const float ar = fabsf(r);
    const float w = ar <= k ? 1.0f : k / ar;
    const float rho = ar <= k ? 0.5f * r * r : k * (ar - 0.5f * k);
    if (res_out) *res_out = r;
    const float wr = w * r;
    sx = fmaf(wr, g0.x, sx);
    sy = fmaf(wr, g0.y, sy);
    acc[kHcE] += rho;
    acc[kHcN] += 1.0f;
}

__device__ __forceinline__ void hc_fold(const PointGeom& G, float sx, float sy, float* acc)
{
    const float v0 = fmaf(sx, G.a0[0], sy * G.a1[0]);
    const float v1 = fmaf(sx, G.a0[1], sy * G.a1[1]);
    const float v2 = fmaf(sx, G.a0[2], sy * G.a1[2]);
    acc[0] += v0;
    acc[1] += v1;
    acc[2] += v2;
    acc[3] += fmaf(G.xr[1], v2, -G.xr[2] * v1);
    acc[4] += fmaf(G.xr[2], v0, -G.xr[0] * v2);
    acc[5] += fmaf(G.xr[0], v1, -G.xr[1] * v0);
}

// Geometric rows at the reference point (identity pose), for the
// inverse-compositional form.
__device__ __forceinline__ void ic_geometry(const StreamDesc& D, const PassParams& P, int p, PointGeom& G)
{
    const float4 q = *checked(D.pt + p, 1, D.pt, (size_t)D.Npad, CK_POINTS);
    const float rho = checked(D.dz + p, 1, D.dz, (size_t)D.Npad, CK_POINTS)->y;
    const float fxl = D.fx * P.scale * rho, fyl = D.fy * P.scale * rho;
    G.a0[0] = fxl;
    G.a0[1] = 0.0f;
    G.a0[2] = -fxl * q.z;
    G.a1[0] = 0.0f;
    G.a1[1] = fyl;
    G.a1[2] = -fyl * q.w;
}

// The p x p patch (the paper's Sec. IV-A patch) for p = 7 and 11, and of any size
// in the cached-Hessian form: the point's
// window of (p + 1) x (p + 1) bytes (inverse compositional) or (p + 3) x (p + 3)
// (forward: the gradient taps) is loaded once with three aligned 8-byte loads
// per row and funnel shifts, and all p*p samples are interpolated from
// registers.  FP32 levels only.
template <int PS, bool ICF, bool HC = false>
__device__ __forceinline__ void linearize_square_t(const StreamDesc& D, const PassParams& P, int p,
                                                   PointGeom& G, float* acc, float* res)
{
    static_assert(!HC || ICF, "the cached Hessian needs the inverse-compositional rows");
    float sx = 0.0f, sy = 0.0f;
    constexpr int h = (PS - 1) / 2, B = ICF ? 0 : 1, R = PS + 1 + 2 * B, NWD = (R + 3) / 4;
    const LevelDev& lv = D.lv[P.level];
    if (ICF) ic_geometry(D, P, p, G);
    const int xs = G.xb - h - B, ys = G.yb - h - B;
    const int a8 = xs & ~7, sh = xs - a8;
    const int wb = sh >> 2, s8 = (sh & 3) * 8;
    const uint8_t* base = lv.img + (size_t)ys * lv.pitch + a8;
    uint32_t win[R][NWD];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint2* rp = checked(reinterpret_cast<const uint2*>(base + (size_t)r * lv.pitch), 3,
                                  reinterpret_cast<const uint2*>(lv.img), (size_t)lv.pitch * lv.H / 8, CK_IMAGE);
        const uint2 u0 = __ldca(rp), u1 = __ldca(rp + 1), u2 = __ldca(rp + 2);
        const uint32_t v[6] = {u0.x, u0.y, u1.x, u1.y, u2.x, u2.y};
#pragma unroll
        for (int i = 0; i < NWD; ++i) {
            const uint32_t lo = wb ? v[i + 1] : v[i];
            const uint32_t hi = wb ? v[i + 2] : v[i + 1];
            win[r][i] = __funnelshift_r(lo, hi, s8);
        }
    }
#define GLT_WX(r, c) u8f(win[(r)][(c) >> 2], (c) & 3)
    constexpr int TG = HC ? hc_groups(PS) : 1;
    // the point's samples of the tables, all groups'
    const size_t from = patch_index<PS, TG>(D, P.level, p, 0, 0), count = (size_t)(group_samples(PS, TG) - 1) * D.Npad * TG + TG;
    const float* I0p = table_from(D, D.I0, from, count);
    const float2* G0p = ICF ? table_from(D, D.G0, from, count) : nullptr;
    const float w00 = (1.0f - G.al) * (1.0f - G.be), w10 = G.al * (1.0f - G.be);
    const float w01 = (1.0f - G.al) * G.be, w11 = G.al * G.be;
#pragma unroll
    for (int j = 0; j < PS; ++j) {
#pragma unroll
        for (int i = 0; i < PS; ++i) {
            const int r0 = j + B, c0 = i + B, k = j * PS + i;
            const size_t at = patch_index<PS, TG>(D, P.level, p, j, i) - from;
            const float i0 = I0p[at];
            const float I00 = GLT_WX(r0, c0), I10 = GLT_WX(r0, c0 + 1);
            const float I01 = GLT_WX(r0 + 1, c0), I11 = GLT_WX(r0 + 1, c0 + 1);
            const float I = fmaf(w00, I00, fmaf(w10, I10, fmaf(w01, I01, w11 * I11)));
            if (HC) {
                hc_sample(I, i0, G0p[at], P.ea, P.b, D.huber_k, sx, sy, acc,
                          res ? res + (size_t)(PS * PS) * p + k : nullptr);
                continue;
            }
            float gx, gy;
            if (ICF) {
                const float2 g0 = G0p[at];
                gx = P.ea * g0.x;
                gy = P.ea * g0.y;
            } else {
                gx = 0.5f * fmaf(w00, I10 - GLT_WX(r0, c0 - 1),
                            fmaf(w10, GLT_WX(r0, c0 + 2) - I00,
                            fmaf(w01, I11 - GLT_WX(r0 + 1, c0 - 1),
                                 w11 * (GLT_WX(r0 + 1, c0 + 2) - I01))));
                gy = 0.5f * fmaf(w00, I01 - GLT_WX(r0 - 1, c0),
                            fmaf(w10, I11 - GLT_WX(r0 - 1, c0 + 1),
                            fmaf(w01, GLT_WX(r0 + 2, c0) - I00,
                                 w11 * (GLT_WX(r0 + 2, c0 + 1) - I10))));
            }
            accumulate_sample(G, I, gx, gy, i0, P.ea, P.b, D.huber_k, acc,
                              res ? res + (size_t)(PS * PS) * p + k : nullptr);
        }
    }
#undef GLT_WX
    if (HC) hc_fold(G, sx, sy, acc);
}

// Any other odd p (3..11) with H summed in every pass: samples read one by one
// (four taps, plus the gradient taps in the forward form).
__device__ __forceinline__ void linearize_square_any(const StreamDesc& D, const PassParams& P, int p,
                                                     PointGeom& G, float* acc, float* res)
{
    const LevelDev& lv = D.lv[P.level];
    const int K = D.K, h = (D.pattern - 1) / 2, S = lv.pitch;
    const bool ic = D.G0 != nullptr;
    if (ic) ic_geometry(D, P, p, G);
    const float w00 = (1.0f - G.al) * (1.0f - G.be), w10 = G.al * (1.0f - G.be);
    const float w01 = (1.0f - G.al) * G.be, w11 = G.al * G.be;
    const size_t from = patch_index1(D, P.level, p, 0), count = (size_t)(K - 1) * D.Npad + 1;
    const float* I0p = table_from(D, D.I0, from, count);
    const float2* G0p = ic ? table_from(D, D.G0, from, count) : nullptr;
    for (int k = 0; k < K; ++k) {
        const size_t at = (size_t)k * D.Npad;
        const float i0 = I0p[at];
        const int dx = k % D.pattern - h, dy = k / D.pattern - h;
        // taps t - S - 1 .. t + 2 S + 2 (intensity and central differences)
        const uint8_t* t = checked(lv.img + (size_t)(G.yb + dy - 1) * S + (G.xb + dx - 1), (size_t)3 * S + 4,
                                   lv.img, (size_t)S * lv.H, CK_IMAGE) + S + 1;
        const float I00 = __ldca(t), I10 = __ldca(t + 1), I01 = __ldca(t + S), I11 = __ldca(t + S + 1);
        const float I = fmaf(w00, I00, fmaf(w10, I10, fmaf(w01, I01, w11 * I11)));
        float gx, gy;
        if (ic) {
            const float2 g0 = G0p[at];
            gx = P.ea * g0.x;
            gy = P.ea * g0.y;
        } else {
            gx = 0.5f * fmaf(w00, I10 - (float)__ldca(t - 1),
                        fmaf(w10, (float)__ldca(t + 2) - I00,
                        fmaf(w01, I11 - (float)__ldca(t + S - 1),
                             w11 * ((float)__ldca(t + S + 2) - I01))));
            gy = 0.5f * fmaf(w00, I01 - (float)__ldca(t - S),
                        fmaf(w10, I11 - (float)__ldca(t - S + 1),
                        fmaf(w01, (float)__ldca(t + 2 * S) - I00,
                             w11 * ((float)__ldca(t + 2 * S + 1) - I10))));
        }
        accumulate_sample(G, I, gx, gy, i0, P.ea, P.b, D.huber_k, acc, res ? res + (size_t)K * p + k : nullptr);
    }
}

// Inlined so the accumulators stay in registers.
template <bool HC = false>
__device__ __forceinline__ void linearize_square(const StreamDesc& D, const PassParams& P, int p,
                                                 PointGeom& G, float* acc, float* res)
{
    if (HC) {
        // (glt_debug_linearize; 9 x 9, 2000 points: 54 us a call, 66 sample by sample)
        switch (D.pattern) {
        case 3: linearize_square_t<3, true, true>(D, P, p, G, acc, res); break;
        case 5: linearize_square_t<5, true, true>(D, P, p, G, acc, res); break;
        case 7: linearize_square_t<7, true, true>(D, P, p, G, acc, res); break;
        case 9: linearize_square_t<9, true, true>(D, P, p, G, acc, res); break;
        default: linearize_square_t<11, true, true>(D, P, p, G, acc, res); break;
        }
        return;
    }
    const bool ic = D.G0 != nullptr;
    if (D.pattern == 7) {
        if (ic) linearize_square_t<7, true>(D, P, p, G, acc, res);
        else linearize_square_t<7, false>(D, P, p, G, acc, res);
    } else if (D.pattern == 11) {
        if (ic) linearize_square_t<11, true>(D, P, p, G, acc, res);
        else linearize_square_t<11, false>(D, P, p, G, acc, res);
    } else {
        linearize_square_any(D, P, p, G, acc, res);
    }
}

// A group of rows of a p x p patch in the cached-Hessian form (TG threads per
// point; TG = 1: the whole patch): each of the point's threads projects the point
// (the same FP32 arithmetic, so the same validity decision), samples its rows
// from its own (rows + 1) x (p + 1) byte window and folds its rows' sums into g0;
// the fold is linear, so the threads of a point exchange nothing.
template <int PS, int TG>
__device__ __forceinline__ void linearize_rows_hc(const StreamDesc& D, const PassParams& P, int p,
                                                  int group, PointGeom& G, float* acc)
{
    constexpr int h = (PS - 1) / 2, RG = group_rows(PS, TG), R = RG + 1;
    constexpr int NWD = (PS + 1 + 3) / 4;
    const LevelDev& lv = D.lv[P.level];
    ic_geometry(D, P, p, G);
    const int j0 = group * RG;
    const int xs = G.xb - h, ys = G.yb - h + j0;
    const int a8 = xs & ~7, sh = xs - a8;
    const int wb = sh >> 2, s8 = (sh & 3) * 8;
    const uint8_t* base = lv.img + (size_t)ys * lv.pitch + a8;
    uint32_t win[R][NWD];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        // rows of the patch (and the lower bilinear tap of its last row) only
        if (j0 + r <= PS) {
            const uint2* rp = checked(reinterpret_cast<const uint2*>(base + (size_t)r * lv.pitch), 3,
                                      reinterpret_cast<const uint2*>(lv.img), (size_t)lv.pitch * lv.H / 8,
                                      CK_IMAGE);
            const uint2 u0 = __ldca(rp), u1 = __ldca(rp + 1), u2 = __ldca(rp + 2);
            const uint32_t v[6] = {u0.x, u0.y, u1.x, u1.y, u2.x, u2.y};
#pragma unroll
            for (int i = 0; i < NWD; ++i) {
                const uint32_t lo = wb ? v[i + 1] : v[i];
                const uint32_t hi = wb ? v[i + 2] : v[i + 1];
                win[r][i] = __funnelshift_r(lo, hi, s8);
            }
        } else {
#pragma unroll
            for (int i = 0; i < NWD; ++i) win[r][i] = 0u;
        }
    }
#define GLT_WR(r, c) u8f(win[(r)][(c) >> 2], (c) & 3)
    const float w00 = (1.0f - G.al) * (1.0f - G.be), w10 = G.al * (1.0f - G.be);
    const float w01 = (1.0f - G.al) * G.be, w11 = G.al * G.be;
    // this task's column of the tables: sample l of the group is l strides on
    const size_t stride = (size_t)D.Npad * TG, at0 = patch_index<PS, TG>(D, P.level, p, j0, 0);
    const size_t count = (size_t)(min(RG, PS - j0) * PS - 1) * stride + 1;
    const float* I0p = table_from(D, D.I0, at0, count);
    const float2* G0p = table_from(D, D.G0, at0, count);
    float sx = 0.0f, sy = 0.0f;
    // UNIT: every residual is within the Huber threshold, so that the weight is 1
    // and the energy r^2 / 2 (hc_sample's operations without the two selects and
    // the division, in its order)
    auto sum = [&](auto unit) {
        constexpr bool UNIT = decltype(unit)::value;
        float E = acc[kHcE];
#pragma unroll
        for (int j = 0; j < RG; ++j) {
            if (j0 + j < PS) {
#pragma unroll
                for (int i = 0; i < PS; ++i) {
                    const size_t at = (j * PS + i) * stride;
                    const float I00 = GLT_WR(j, i), I10 = GLT_WR(j, i + 1);
                    const float I01 = GLT_WR(j + 1, i), I11 = GLT_WR(j + 1, i + 1);
                    const float I = fmaf(w00, I00, fmaf(w10, I10, fmaf(w01, I01, w11 * I11)));
                    const float i0 = I0p[at];
                    const float2 g0 = G0p[at];
                    if (UNIT) {
                        const float r = __fsub_rn(fmaf(-P.ea, i0, I), P.b);
                        sx = fmaf(r, g0.x, sx);
                        sy = fmaf(r, g0.y, sy);
                        E = __fadd_rn(E, __fmul_rn(__fmul_rn(0.5f, r), r));
                    } else {
                        hc_sample(I, i0, g0, P.ea, P.b, D.huber_k, sx, sy, acc, nullptr);
                    }
                }
            }
        }
        if (UNIT) {
            acc[kHcE] = E;
            acc[kHcN] += (float)(min(RG, PS - j0) * PS);
        }
    };
    // |r| <= 255 (1 + e^a) + |b| and a few roundings.  The paper's own
    // configuration has no threshold: its 66 passes take 339 us with UNIT, 437
    // without (2000 points, 7 x 7), 438 and 700 at 11 x 11
    if (fmaf(P.ea, 256.0f, 256.0f) + 1.001f * fabsf(P.b) <= D.huber_k)
        sum(std::true_type{});
    else
        sum(std::false_type{});
#undef GLT_WR
    hc_fold(G, sx, sy, acc);
}

// Linearises map point p at the pass state into acc.  RES: also write the K
// residuals (NaN for an unusable point) to res[Kp..Kp+K-1].
// SQUARE: the p x p path is compiled in; IC: the inverse-compositional rows
// are compiled in (both decided per stream at run time when compiled in).
// HC: the cached-Hessian accumulation (acc holds kHcAcc values; FP32 levels
// and inverse-compositional rows only).
template <bool MIXED, bool RES, bool SQUARE = false, bool IC = true, bool HC = false>
__device__ __forceinline__ void linearize_point(const StreamDesc& D, const PassParams& P,
                                                const PointCache& c, float* acc, float* res)
{
    static_assert(!HC || (IC && !MIXED), "the cached Hessian needs FP32 levels and IC rows");
    const LevelDev& lv = D.lv[P.level];
    const int p = c.p;
    const float4 ia = c.ia, ib = c.ib;
    PointGeom G;
    bool ok = !isnan(ia.x) && project_point<SQUARE>(D, P, lv, c, G);
    if (!ok) {
        if (RES) {
            for (int k = 0; k < D.K; ++k) res[(size_t)D.K * p + k] = __int_as_float(0x7fc00000);
        }
        return;
    }
    if (SQUARE && D.pattern) {
        linearize_square<HC>(D, P, p, G, acc, RES ? res : nullptr);
        return;
    }
    const float i0[8] = {ia.x, ia.y, ia.z, ia.w, ib.x, ib.y, ib.z, ib.w};
    // inverse-compositional form: geometric rows at the reference point
    // (identity pose) and the cached reference gradients times e^a
    const bool ic = IC && D.G0 != nullptr;
    const float2* G0p = nullptr;
    if (ic) {
        ic_geometry(D, P, p, G);
        G0p = checked(D.G0 + ((size_t)P.level * D.Npad + p) * 8, (size_t)8, D.G0, (size_t)D.L * D.Npad * 8,
                      CK_TABLE);
    }
    const float w00 = (1.0f - G.al) * (1.0f - G.be), w10 = G.al * (1.0f - G.be);
    const float w01 = (1.0f - G.al) * G.be, w11 = G.al * G.be;
    if (!MIXED) {
        // 8x8 byte window, rows yb-3..yb+4, columns xb-3..xb+4: two aligned
        // 8-byte loads per row, those that hold a byte of the row in use (12 of 16
        // on average: every lane's load is a tag lookup of its own), then a funnel
        // shift to the window start.
        float hsx = 0.0f, hsy = 0.0f;   // cached-Hessian form: the point's (sx, sy)
        const int xs = G.xb - 3;
        const int a8 = xs & ~7;
        const int off = xs - a8, sh = off * 8;
        const bool far = sh >= 32;
        const uint8_t* base = lv.img + (size_t)(G.yb - 3) * lv.pitch + a8;
        uint32_t rw[8][2];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint2* rp = checked(reinterpret_cast<const uint2*>(base + (size_t)r * lv.pitch), 2,
                                      reinterpret_cast<const uint2*>(lv.img), (size_t)lv.pitch * lv.H / 8,
                                      CK_IMAGE);
            const int lo = r < 4 ? 3 - r : r - 4, hi = 7 - lo;      // the row's columns of the pattern and its gradients
            const uint2 w0 = off + lo < 8 ? __ldca(rp) : make_uint2(0u, 0u), w1 = off + hi >= 8 ? __ldca(rp + 1) : make_uint2(0u, 0u);
            const uint32_t v0 = far ? w0.y : w0.x, v1 = far ? w1.x : w0.y, v2 = far ? w1.y : w1.x;
            rw[r][0] = __funnelshift_r(v0, v1, sh);      // (by sh modulo 32)
            rw[r][1] = __funnelshift_r(v1, v2, sh);
        }
#define GLT_PX(r, c) u8f(rw[(r)][(c) >> 2], (c) & 3)
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int r0 = pat_dy(k) + 3, c0 = pat_dx(k) + 3;
            const float I00 = GLT_PX(r0, c0), I10 = GLT_PX(r0, c0 + 1);
            const float I01 = GLT_PX(r0 + 1, c0), I11 = GLT_PX(r0 + 1, c0 + 1);
            const float I = fmaf(w00, I00, fmaf(w10, I10, fmaf(w01, I01, w11 * I11)));
            if (HC) {
                hc_sample(I, i0[k], G0p[k], P.ea, P.b, D.huber_k, hsx, hsy, acc,
                          RES ? res + 8 * p + k : nullptr);
                continue;
            }
            float gx, gy;
            if (ic) {
                const float2 g0 = G0p[k];
                gx = P.ea * g0.x;
                gy = P.ea * g0.y;
            } else {
                // central differences at the four taps (the 1/2 is applied after interpolation)
                gx = 0.5f * fmaf(w00, I10 - GLT_PX(r0, c0 - 1),
                            fmaf(w10, GLT_PX(r0, c0 + 2) - I00,
                            fmaf(w01, I11 - GLT_PX(r0 + 1, c0 - 1),
                                 w11 * (GLT_PX(r0 + 1, c0 + 2) - I01))));
                gy = 0.5f * fmaf(w00, I01 - GLT_PX(r0 - 1, c0),
                            fmaf(w10, I11 - GLT_PX(r0 - 1, c0 + 1),
                            fmaf(w01, GLT_PX(r0 + 2, c0) - I00,
                                 w11 * (GLT_PX(r0 + 2, c0 + 1) - I10))));
            }
            accumulate_sample<false>(G, I, gx, gy, i0[k], P.ea, P.b, D.huber_k, acc,
                              RES ? res + 8 * p + k : nullptr);
        }
#undef GLT_PX
        if (HC)
            hc_fold(G, hsx, hsy, acc);
        else
            acc[kIdxN] += 8.0f;
    } else {
        const uint2* pk = lv.packed;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int x0 = G.xb + pat_dx(k), y0 = G.yb + pat_dy(k);
            const uint2* t0 = checked(pk + (size_t)y0 * lv.W + x0, (size_t)lv.W + 2, pk, (size_t)lv.W * lv.H,
                                      CK_PACKED);
            const uint2* t1 = t0 + lv.W;
            const uint2 p00 = __ldca(t0), p10 = __ldca(t0 + 1), p01 = __ldca(t1), p11 = __ldca(t1 + 1);
            const float2 a00 = __half22float2(*reinterpret_cast<const __half2*>(&p00.x));
            const float2 a10 = __half22float2(*reinterpret_cast<const __half2*>(&p10.x));
            const float2 a01 = __half22float2(*reinterpret_cast<const __half2*>(&p01.x));
            const float2 a11 = __half22float2(*reinterpret_cast<const __half2*>(&p11.x));
            const float y00 = __low2float(*reinterpret_cast<const __half2*>(&p00.y));
            const float y10 = __low2float(*reinterpret_cast<const __half2*>(&p10.y));
            const float y01 = __low2float(*reinterpret_cast<const __half2*>(&p01.y));
            const float y11 = __low2float(*reinterpret_cast<const __half2*>(&p11.y));
            const float I = fmaf(w00, a00.x, fmaf(w10, a10.x, fmaf(w01, a01.x, w11 * a11.x)));
            const float2 g0 = ic ? G0p[k] : make_float2(0.0f, 0.0f);
            const float gx = ic ? P.ea * g0.x : fmaf(w00, a00.y, fmaf(w10, a10.y, fmaf(w01, a01.y, w11 * a11.y)));
            const float gy = ic ? P.ea * g0.y : fmaf(w00, y00, fmaf(w10, y10, fmaf(w01, y01, w11 * y11)));
            accumulate_sample<false>(G, I, gx, gy, i0[k], P.ea, P.b, D.huber_k, acc,
                              RES ? res + 8 * p + k : nullptr);
        }
        acc[kIdxN] += 8.0f;
    }
}

// One task of a cached-Hessian pass: row group `group` of point c.p for the
// 7 x 7 and 11 x 11 patches, the whole point otherwise (group = 0).
__device__ __forceinline__ void linearize_task_hc(const StreamDesc& D, const PassParams& P,
                                                  const PointCache& c, int group, float* acc)
{
    if (!D.pattern) {
        linearize_point<false, false, false, true, true>(D, P, c, acc, nullptr);
        return;
    }
    const LevelDev& lv = D.lv[P.level];
    PointGeom G;
    if (isnan(c.ia.x) || !project_point<true>(D, P, lv, c, G)) return;
    switch (D.pattern) {
    case 3: linearize_rows_hc<3, 1>(D, P, c.p, 0, G, acc); break;
    case 5: linearize_rows_hc<5, 1>(D, P, c.p, 0, G, acc); break;
    case 7: linearize_rows_hc<7, kHcGroups>(D, P, c.p, group, G, acc); break;
    case 9: linearize_rows_hc<9, 1>(D, P, c.p, 0, G, acc); break;
    default: linearize_rows_hc<11, kHcGroups>(D, P, c.p, group, G, acc); break;
    }
}

// ---------------------------------------------------------------------------
// Reductions
// ---------------------------------------------------------------------------
// Butterfly reduce-scatter of 48 values over a warp: 48 shuffles instead of
// 5 x 48.  Afterwards lane L holds the warp sums of indices
// base(L) + {0,1,2}, base = 24*b4 + 12*b3 + 6*b2 + 3*b1 (b_i = bit i of L).
__device__ __forceinline__ int rs_base(int lane)
{
    return ((lane >> 4) & 1) * 24 + ((lane >> 3) & 1) * 12 + ((lane >> 2) & 1) * 6 + ((lane >> 1) & 1) * 3;
}

__device__ __forceinline__ void warp_reduce_scatter48(float (&v)[kAccPad], int lane)
{
    const unsigned full = 0xffffffffu;
#define GLT_RS_STAGE(HALF, OFF)                                            \
    {                                                                      \
        const bool hi = (lane & (OFF)) != 0;                               \
        _Pragma("unroll") for (int i = 0; i < (HALF); ++i) {               \
            const float send = hi ? v[i] : v[i + (HALF)];                  \
            const float keep = hi ? v[i + (HALF)] : v[i];                  \
            v[i] = keep + __shfl_xor_sync(full, send, (OFF));              \
        }                                                                  \
    }
    GLT_RS_STAGE(24, 16)
    GLT_RS_STAGE(12, 8)
    GLT_RS_STAGE(6, 4)
    GLT_RS_STAGE(3, 2)
#undef GLT_RS_STAGE
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] += __shfl_xor_sync(full, v[i], 1);
}

// Butterfly reduce-scatter of the 8 cached-Hessian accumulators (7 shuffles),
// then two pair stages: afterwards lanes with (lane & 3) == 0 hold the warp
// sum of value ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1).
__device__ __forceinline__ int rs8_index(int lane)
{
    return ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
}

__device__ __forceinline__ void warp_reduce_scatter8(float (&v)[kHcAcc], int lane)
{
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int half = 4, off = 16; half >= 1; half >>= 1, off >>= 1) {
        const bool hi = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = hi ? v[i] : v[i + half];
            const float keep = hi ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(full, send, off);
        }
    }
    v[0] += __shfl_xor_sync(full, v[0], 2);
    v[0] += __shfl_xor_sync(full, v[0], 1);
}

// Block reduction of the 8 cached-Hessian accumulators into out[0..8).
// Ends with __syncthreads().
template <int THREADS>
__device__ __forceinline__ void block_reduce8(float (&acc)[kHcAcc], float (*red)[kAccPad], float* out)
{
    constexpr int NW = THREADS / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    warp_reduce_scatter8(acc, lane);
    if ((lane & 3) == 0) red[warp][rs8_index(lane)] = acc[0];
    __syncthreads();
    if (threadIdx.x < kHcAcc) {
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) s += red[w][threadIdx.x];
        out[threadIdx.x] = s;
    }
    __syncthreads();
}

// Block reduction of the per-thread accumulators into out[0..kNumAcc).
// KAHAN: compensated FP32 sum across warps, compensation in out_c.
// Ends with __syncthreads().
template <int THREADS, bool KAHAN>
__device__ __forceinline__ void block_reduce(float (&acc)[kAccPad], float (*red)[kAccPad], float* out,
                                             float* out_c)
{
    constexpr int NW = THREADS / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    warp_reduce_scatter48(acc, lane);
    if ((lane & 1) == 0) {
        const int b = rs_base(lane);
        red[warp][b + 0] = acc[0];
        red[warp][b + 1] = acc[1];
        red[warp][b + 2] = acc[2];
    }
    __syncthreads();
    if (threadIdx.x < kNumAcc) {
        const int j = threadIdx.x;
        float s = 0.0f, c = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            if (KAHAN) {
                const float y = red[w][j] - c;
                const float t = s + y;
                c = (t - s) - y;
                s = t;
            } else {
                s += red[w][j];
            }
        }
        out[j] = s;
        if (KAHAN) out_c[j] = -c;
    }
    __syncthreads();
}

// f as a double, in integers: the conversion would hold the FP64 pipe for 64
// cycles, as long as the addition that follows it.
__device__ __forceinline__ double exact_double(float f)
{
    const unsigned u = __float_as_uint(f), sign = u & 0x80000000u;
    unsigned m = u & 0x7fffffffu, off = 0x38000000u;           // exponent bias 1023 - 127
    if (m >= 0x7f800000u) off = 0x70000000u;                   // infinities, NaN
    if (m < 0x00800000u) {                                     // zero, subnormals: normalised
        const int lz = m ? __clz((int)m) - 8 : 0;
        off = m ? 0x38100000u - ((unsigned)lz << 20) : 0u;
        m = (m << lz) & 0x7fffffu;
    }
    return __hiloint2double((int)(sign | ((m >> 3) + off)), (int)(m << 29));
}

// Sums of the blocks' partials [blocks][kAccPad] in FP64, by the last block of a
// linearisation: 10 interleaved chains of sum_cols(NSUM) / 4 threads with four
// sums each, eight loads in flight a thread.  A block stores sum_cols(NSUM)
// columns, zeros beyond its NSUM sums.  Bound by the FP64 additions, 64 cycles
// each on the four pipes of the SM: 10.7k cycles for 46 sums of 157 blocks, 19.8k
// with one chain per sum and a load at a time.
__host__ __device__ constexpr int sum_cols(int nsum) { return (nsum + 3) / 4 * 4; }

template <int NSUM, int THREADS>
__device__ __forceinline__ void sum_partials(const float* partials, unsigned blocks, double* out)
{
    constexpr int QUADS = sum_cols(NSUM) / 4, CHAINS = 10, AHEAD = 8;
    static_assert(QUADS * CHAINS <= THREADS && NSUM <= THREADS && sum_cols(NSUM) <= kAccPad, "a thread per quad of a chain and per sum");
    __shared__ double red[CHAINS][kAccPad];
    const int t = threadIdx.x, q = t % QUADS, chain = t / QUADS;
    if (chain < CHAINS) {
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        for (unsigned b0 = chain; b0 < blocks; b0 += AHEAD * CHAINS) {
            float4 v[AHEAD];
#pragma unroll
            for (int k = 0; k < AHEAD; ++k) {
                const unsigned b = b0 + k * CHAINS;
                v[k] = b < blocks ? __ldcg(reinterpret_cast<const float4*>(partials + (size_t)b * kAccPad) + q)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int k = 0; k < AHEAD; ++k) {
                if (b0 + k * CHAINS >= blocks) break;
                s[0] += exact_double(v[k].x);
                s[1] += exact_double(v[k].y);
                s[2] += exact_double(v[k].z);
                s[3] += exact_double(v[k].w);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) red[chain][4 * q + i] = s[i];
    }
    __syncthreads();
    if (t < NSUM) {
        double s = red[0][t];
        for (unsigned c = 1; c < CHAINS && c < blocks; ++c) s += red[c][t];
        out[t] = s;
    }
}

// ---------------------------------------------------------------------------
// Solver tail, run by one warp of every CTA
//
// It sits on the critical path of every pass, and GB300's FP64 is what bounds
// it: measured on the part, an FP64 instruction occupies its sub-partition's
// pipe for 64 cycles whether 1 or 32 lanes take part; the next FP64
// instruction has its result after the same 64, any other after ~110, an
// FP64 compare costs ~105; a shuffle costs ~24 and an FP32 FMA 4.  So the tail
// is written for the fewest FP64 instructions on the dependent chain:
// independent quantities share one instruction on different lanes, comparisons
// go through the bit pattern, and what a decision does not need is not computed.  The state, the normal
// equations, the accept/reject decision and the composition are FP64 in both
// solve modes; GLT_SOLVE_FP64 (the default) also factorises and exponentiates
// in FP64, GLT_SOLVE_FP32 does those two in FP32 (their inputs carry FP32
// rounding anyway, or their result is a small increment):
//  * the damped normal matrix is factored as L D L^T (no square roots), one
//    entry per lane, columns eliminated right-looking with warp shuffles; in
//    GLT_SOLVE_FP32 first in FP32, and a pivot below 1e-4 of its damped
//    diagonal sends the system to the FP64 elimination, which alone decides
//    "not positive definite";
//  * FP64 pivot reciprocals are an FP32 seed and one Newton step in 64-bit
//    integers (rcp_mid);
//  * the SE(3) exponential uses the power series of its coefficients in
//    theta^2 below theta = 0.1 (sincos only beyond), each lane one element
//    of exp(delta) (GLT_SOLVE_FP32: of exp(delta) - I in FP32, composed with
//    the FP64 pose as T + T (exp(delta) - I), and the frame's final pose
//    orthonormalised once in FP64);
//  * accept/reject compares E' n <= E n' instead of dividing, and only for
//    steps that are not small enough to be taken anyway.
// ---------------------------------------------------------------------------
// 1 / d for a positive d in [2^-100, 2^100) without an FP64 instruction: one
// Newton step in integers.  With d = 2^E m, m = M / 2^52 in [1, 2), the seed q =
// rcp.approx.ftz.f32 of m cut to FP32 is Q / 2^24 with a whole Q; the residual e
// = 1 - m q, at most 2^-22, is exactly -(M Q) modulo 2^64 in units of 2^-76, and
// q + q e is formed on the bits of the result (units of 2^-53) and lowered by E
// in the exponent.  The value of r0 + r0 (1 - d r0) in FP64 to an ulp (relative
// error e^2 < 2^-43.9 and that ulp), without its two dependent FP64 instructions
// (128 cycles) and their way out of the FP64 pipe.
__device__ __forceinline__ double rcp_mid(double d)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    float q;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(__uint_as_float((__funnelshift_l(lo, hi, 3) & 0x7fffffu) | 0x3f800000u)));
    const unsigned qb = __float_as_uint(q);
    const unsigned Q = qb >= 0x3f800000u ? 0x1000000u : (qb & 0x7fffffu) | 0x800000u;
    const unsigned long long M = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const long long e = -(long long)(M * Q);
    const int es = (int)((e + (1ll << 23)) >> 24);
    const long long c = ((long long)es * (int)Q + (1ll << 22)) >> 23;
    const unsigned off = ((896u + 1023u) << 20) - (hi & 0x7ff00000u);
    return __longlong_as_double(((long long)qb << 29) + c + ((long long)off << 32));
}

// Reciprocal of any d: rcp_mid for 2^-100 <= |d| < 2^100 (exponent tested as
// an integer); zero, infinities, NaN and the rest divide.
__device__ __forceinline__ double rcp_d(double d)
{
    const int ebits = (__double2hiint(d) >> 20) & 0x7ff;
    if (ebits < 1023 - 100 || ebits >= 1023 + 100) return 1.0 / d;
    return copysign(rcp_mid(fabs(d)), d);
}

// FP64 -> FP32 through the bit pattern (integer instructions only, nothing on
// the FP64 pipe): the significand truncated to 23 bits (relative error
// < 2^-23); magnitudes below 2^-126 give a signed zero and above FP32's range
// infinity; infinities and NaN are kept.
__device__ __forceinline__ float f32_of(double x)
{
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const int eb = (hi >> 20) & 0x7ff;
    const unsigned sign = (unsigned)hi & 0x80000000u;
    const unsigned man = (((unsigned)hi & 0xfffffu) << 3) | (lo >> 29);
    unsigned b;
    if (eb == 0x7ff)
        b = sign | 0x7f800000u | ((((unsigned)hi & 0xfffffu) | lo) ? 0x400000u : 0u);
    else if (eb > 1023 + 127)
        b = sign | 0x7f800000u;
    else if (eb < 1023 - 126)
        b = sign;
    else
        b = sign | ((unsigned)(eb - 896) << 23) | man;
    return __uint_as_float(b);
}

// FP64 -> FP32 rounded to nearest even, as the conversion instruction does it,
// in integer instructions (the conversion takes its turn on the FP64 pipe), for
// finite x; magnitudes below FP32's normal range give a signed zero.
__device__ __forceinline__ float f32_rn(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned eb = (hi >> 20) & 0x7ffu;
    // re-biased exponent, 23 bits of the significand; a carry out of the
    // rounded significand steps the exponent
    unsigned b = (__funnelshift_l(lo, hi, 3) & 0x7fffffu) | ((eb - 896u) << 23);
    const unsigned rem = lo << 3;                  // what the cut leaves, 2^31 is half
    if (rem > 0x80000000u - (b & 1u)) ++b;
    if (eb < 897u) b = 0u;
    if (eb > 1150u) b = 0x7f800000u;
    return __uint_as_float(b | (hi & 0x80000000u));
}

// FP32 -> FP64 through the bit pattern: exact for zero and normal numbers
// (subnormals give a signed zero); infinities and NaN are kept.
__device__ __forceinline__ double f64_of(float f)
{
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xffu;
    const unsigned sign = b & 0x80000000u;
    unsigned hi = sign, lo = 0u;
    if (e != 0u) {
        hi = sign | ((e == 0xffu ? 0x7ffu : e + 896u) << 20) | ((b & 0x7fffffu) >> 3);
        if (e == 0xffu && (b & 0x7fffffu)) hi |= 0x80000u;
        lo = b << 29;
    }
    return __hiloint2double((int)hi, (int)lo);
}

// |x| compared through the bit pattern: for non-negative doubles the IEEE
// ordering is the integer ordering of the bits (no FP64 instructions).
__device__ __forceinline__ long long abs_bits(double x)
{
    return __double_as_longlong(x) & 0x7fffffffffffffffll;
}

// Bits of +infinity: x is finite iff abs_bits(x) < kInfBits.
constexpr long long kInfBits = 0x7ff0000000000000ll;

// Pass parameters for state (T, a, b) on `level` (single thread).
__device__ __host__ inline void make_pass_params(const double* T, double a, double b, int level,
                                                 PassParams& P)
{
    P.Rm[0] = (float)(T[0] - 1.0);
    P.Rm[1] = (float)T[1];
    P.Rm[2] = (float)T[2];
    P.Rm[3] = (float)T[4];
    P.Rm[4] = (float)(T[5] - 1.0);
    P.Rm[5] = (float)T[6];
    P.Rm[6] = (float)T[8];
    P.Rm[7] = (float)T[9];
    P.Rm[8] = (float)(T[10] - 1.0);
    P.t[0] = (float)T[3];
    P.t[1] = (float)T[7];
    P.t[2] = (float)T[11];
    P.ea = expf((float)a);
    P.b = (float)b;
    P.level = level;
    P.scale = ldexpf(1.0f, -level);
    P.done = 0;
}

// Same, one element per lane (lanes 0-13), for the pose in T (12 doubles).
__device__ __forceinline__ void make_pass_params_warp(const double* T, double a, double b,
                                                      int level, PassParams& P, int lane)
{
    if (lane < 12) {
        const int r = lane >> 2, c = lane & 3;
        const double v = T[lane] - ((c == r) ? 1.0 : 0.0);
        if (c < 3)
            P.Rm[3 * r + c] = (float)v;
        else
            P.t[r] = (float)v;
    } else if (lane == 12) {
        P.ea = expf((float)a);
    } else if (lane == 13) {
        P.b = (float)b;
        P.level = level;
        P.scale = ldexpf(1.0f, -level);
        P.done = 0;
    }
}

// Constants behind the two states and behind the step, so that a lane fetches
// every operand by index (no selects, no divergence).
constexpr int kSt0 = 14, kSt1 = 15, kStM1 = 16, kStDown = 17, kStUp = 18, kStSize = 20;
constexpr int kXs0 = 8, kXs1 = 9, kXsPoly = 10, kXsSize = 20;

// w.w: the state machine's flags
constexpr int kFlCur = 1;      // which state is the accepted one
constexpr int kFlAcc = 2;      // which sums are the accepted state's
constexpr int kFlCand = 4;     // phase: the pass evaluates a candidate
constexpr int kFlSmall = 8;    // the candidate's step is below accept_step
constexpr int kFlStop = 16;    // ... below the level's stop threshold
constexpr int kFlMoved = 32;   // the pose changed since the initial state
constexpr int kFlLevel = 8;    // the level, from this bit on

// LM state machine, replicated in every CTA of a stream's cluster (each CTA
// runs it on bit-identical inputs, so all take the same decisions).
struct Solver {
    // two states [T (12), a, b, then the constants 0, 1, -1 and the damping
    // factors]: the accepted one and the candidate under evaluation
    double st[2][kStSize];
    // two sets of sums: the accepted state's and the last pass's (zeros from
    // kNumAcc on); n[]: their sample counts as integers
    double tot[2][kAccPad];
    double xs[kXsSize];       // the step (translation, rotation, da, db), then 0, 1 and the
                              // series of A, B, C (tail_map_init)
    double Lm[72];            // L row by row, then D^-1 L^-1 times the right-hand side
    double Hi[36];            // cached-Hessian form: -e^-a H^-1 of the level
    double lam[2];            // the damping after the candidate is accepted / rejected
    double ema;               // cached-Hessian form: e^-a (a is held fixed there)
    double res_E;
    int4 w;                   // iterations of the level, status, passes, flags
    int n[2], bad;            // bad: a sum of the last pass is not finite
    int hc_ok;                // the level's reference Hessian is positive definite
    int res_n;
    int iters[kMaxLevels];
    unsigned map_ldl[32], map_dot[32], map_ent[32], map_cmp[32];   // per lane (tail_map_init)
};

// Upper-triangle index of (i, j), i <= j, in the accumulator layout.
__host__ __device__ __forceinline__ constexpr int upper_index(int i, int j) { return i * 8 - (i * (i - 1)) / 2 + (j - i); }

// The sums' buffer a pass writes, and one finished sum (of n samples) into it.
__device__ __forceinline__ int solver_buffer(const Solver& S) { return (S.w.w & kFlAcc) ? 0 : 1; }

template <bool HC>
__device__ __forceinline__ void solver_put_sum(Solver& S, int wb, int i, double v, int n)
{
    S.tot[wb][i] = v;
    // sums that are not finite (an FP32 overflow) make the pass unusable
    if (!(abs_bits(v) < kInfBits)) S.bad = 1;
    if (i == (HC ? kHcN : kIdxN)) S.n[wb] = n;
}

// Initial state (one thread): Gram-Schmidt the initial rotation, first level.
__device__ inline void solver_init(const StreamDesc& D, const double* init, Solver& S, PassParams& P)
{
    double* T = S.st[0];
    for (int i = 0; i < 14; ++i) T[i] = init[i];
    {
        const double n0 = sqrt(T[0] * T[0] + T[1] * T[1] + T[2] * T[2]);
        for (int c = 0; c < 3; ++c) T[c] /= n0;
        const double d = T[4] * T[0] + T[5] * T[1] + T[6] * T[2];
        for (int c = 0; c < 3; ++c) T[4 + c] -= d * T[c];
        const double n1 = sqrt(T[4] * T[4] + T[5] * T[5] + T[6] * T[6]);
        for (int c = 0; c < 3; ++c) T[4 + c] /= n1;
        T[8] = T[1] * T[6] - T[2] * T[5];
        T[9] = T[2] * T[4] - T[0] * T[6];
        T[10] = T[0] * T[5] - T[1] * T[4];
    }
    for (int k = 0; k < 2; ++k) {
        S.st[k][kSt0] = 0.0;
        S.st[k][kSt1] = 1.0;
        S.st[k][kStM1] = -1.0;
        S.st[k][kStDown] = D.lambda_down;
        S.st[k][kStUp] = D.lambda_up;
    }
    int status = 0;
    bool finite_start = true;
    for (int i = 0; i < 14; ++i) finite_start &= abs_bits(T[i]) < kInfBits;
    S.n[0] = S.n[1] = 0;
    S.bad = 0;
    S.res_n = 0;
    S.res_E = __longlong_as_double(0x7ff8000000000000ll);
    for (int l = 0; l < kMaxLevels; ++l) S.iters[l] = 0;
    S.ema = (D.Hc && finite_start) ? exp(-T[12]) : 1.0;
    int l = D.L - 1;
    while (l >= 0 && D.max_iters[l] <= 0) --l;
    if (!finite_start) {
        // a start that is not finite (or whose rotation is degenerate) is
        // not solved: the result is the start, flagged
        status |= GLT_TRACK_DIVERGED;
        l = -1;
    }
    S.w = make_int4(0, status, 0, (l < 0 ? 0 : l) << kFlLevel);
    if (l < 0)
        P.done = 1;
    else
        make_pass_params(T, T[12], T[13], l, P);
}

// Per-lane tables of the tail, packed, and its constants (one warp, once per
// launch; the caller synchronises).
__host__ __device__ constexpr int ldl_lane(int k) { return k == 2 ? 0 : k == 3 ? 7 : k == 4 ? 13 : k == 5 ? 18 : k == 6 ? 22 : 25; }

__device__ inline void tail_map_init(Solver& S, int lane)
{
    // L D L^T: positions of the lane's entries in the sums, and (i, k) of both
    const int kA = lane < 7 ? 2 : lane < 13 ? 3 : lane < 18 ? 4 : lane < 22 ? 5 : lane < 25 ? 6 : lane < 27 ? 7 : 8;
    const int iA = kA < 8 ? kA + lane - ldl_lane(kA) : 9;
    const int kB = lane < 9 ? 0 : lane < 17 ? 1 : 8;
    const int iB = lane < 9 ? lane : lane < 17 ? lane - 8 : 9;
    const int pA = iA > 8 ? kNumAcc : iA == 8 ? kIdxG + kA : upper_index(kA, iA);   // kNumAcc: a zero
    const int pB = iB > 8 ? kNumAcc : iB == 8 ? kIdxG + kB : upper_index(kB, iB);
    S.map_ldl[lane] = (unsigned)(pA | (pB << 6) | (iA << 12) | (kA << 16) | (iB << 20) | (kB << 24));
    // the three products of a lane's dot (indices into xs): w . w on lanes
    // 0-15, w . v on 16, (w x v)_r on 17 + r (its second product negated)
    const int r = lane >= 17 && lane < 20 ? lane - 17 : 0, r1 = (r + 1) % 3, r2 = (r + 2) % 3;
    const bool dot = lane == 16, cross = lane >= 17 && lane < 20;
    const int p1 = cross ? 3 + r1 : 3, q1 = cross ? r2 : dot ? 0 : 3;
    const int p2 = cross ? 3 + r2 : 4, q2 = cross ? r1 : dot ? 1 : 4;
    const int p3 = cross ? kXs0 : 5, q3 = cross ? kXs0 : dot ? 2 : 5;
    S.map_dot[lane] = (unsigned)(p1 | (q1 << 5) | (p2 << 10) | (q2 << 15) | (p3 << 20) | (q3 << 25));
    // entry (er, ec) of the exponential on lane 4 er + ec < 12: w_er, the
    // column's w (rotation), d_rc or v_er, and W_rc = +w_{r+2} if c = r+1 (bit
    // 25: negated), w_{r+1} if c = r+2; lanes 12-14: the series of A, B, C
    const int q = lane & 15, er = (q >> 2) % 3, ec = q & 3, er1 = (er + 1) % 3, er2 = (er + 2) % 3;
    const bool poly = lane >= 12 && lane < 15, rot = ec < 3;
    const int g = lane - 12;
    const int w = poly ? kXsPoly + 6 + g : 3 + er;
    const int pq = poly ? kXs1 : rot ? 3 + ec : kXs0;
    const int dd = poly ? kXsPoly + g : rot ? (er == ec ? kXs1 : kXs0) : er;
    const int c1 = poly ? kXsPoly + 3 + g : kXs0;
    const int W = ec == er1 ? 3 + er2 : (rot && ec == er2) ? 3 + er1 : kXs0;
    S.map_ent[lane] = (unsigned)(w | (pq << 5) | (dd << 10) | (c1 << 15) | (W << 20)) | (ec == er1 ? 1u << 25 : 0u);
    // the composition (indices into a state): row er of T on lanes 4 er + ec
    // and 16 + 4 er + ec, the addend (translation, or minus the identity on
    // lanes 0-11), 1 x da + a, 1 x db + b and the dampings on lanes 12-15
    const int t0 = q < 12 ? 4 * er : kSt0, t1 = q < 12 ? 4 * er + 1 : kSt0;
    const int t2 = q < 12 ? 4 * er + 2 : lane == 12 || lane == 13 ? kSt1 : lane == 14 ? kStDown : lane == 15 ? kStUp : kSt0;
    const int add = q < 12 ? (!rot ? 4 * er + 3 : lane < 12 && er == ec ? kStM1 : kSt0) : lane == 12 || lane == 13 ? lane : kSt0;
    const int pp = lane < 12 ? (rot ? 3 * er + ec : 9 + er) : lane < 14 ? lane : 0;   // entry of P
    S.map_cmp[lane] = (unsigned)(t0 | (t1 << 5) | (t2 << 10) | (add << 15) | (pp << 20));
    if (lane == 0) {
        S.xs[kXs0] = 0.0;
        S.xs[kXs1] = 1.0;
        double* c = S.xs + kXsPoly;      // th^2 coefficients 2 (negated), 1, 0 of A, B, C
        c[0] = -1.0 / 120.0;
        c[1] = -1.0 / 720.0;
        c[2] = -1.0 / 5040.0;
        c[3] = -1.0 / 6.0;
        c[4] = -1.0 / 24.0;
        c[5] = -1.0 / 120.0;
        c[6] = 1.0;
        c[7] = 0.5;
        c[8] = 1.0 / 6.0;
    }
    for (int i = lane; i < 2 * kAccPad; i += 32) (&S.tot[0][0])[i] = 0.0;
}

// -x where `on`, through the sign bit, so that neither an FP64 instruction nor a
// select joins the chain (with the selects of the exponential gone too and a
// shorter pivot test: 7.2k -> 6.9k cycles a tail)
__device__ __forceinline__ double flip_sign(double x, bool on)
{
    return __hiloint2double(__double2hiint(x) ^ (on ? (int)0x80000000 : 0), __double2loint(x));
}

// (H + lambda diag H) delta = -g by L D L^T, right-looking, one entry per
// lane.  The right-hand side rides along as row 8 of the lower triangle
// (entry (8, k) = y_k), so the 44 entries (i, k), k <= i <= 8, all follow
//   a_ik -= a_ij a_kj / d_j   for k > j.
// Columns 2-7 (27 entries) sit in register A of lanes 0-26 and take one FMA
// per eliminated column; columns 0 and 1 sit in register B of lanes 0-8 and
// 9-16, of which column 1 is updated once.  Column k starts at lane cA(k) of
// A, so entry (i, j) is on lane cA(j) - j + i (B: i for j = 0, 8 + i for j =
// 1); a lane without part in a step takes its factors from lane 31, which
// holds zeros.  The product a_ij a_kj is formed while the pivot's reciprocal
// is, so a column's dependent chain is a shuffle, the product and one FMA.
// (With l_ij = a_ij / d_j, a Newton step in FP64 and separate updates of the
// diagonal and the right-hand side the solve took 6.9k cycles.)
// tot: a pass's sums (zeros beyond the last); Lm: 72 doubles of shared memory;
// x: the solution on lanes 0-7.  EXACT: reciprocals of any pivot and the pivot
// test d > 0, d > 1e-13 x the damped diagonal; otherwise every pivot must
// pass that test by its exponent alone (2^-43 > 1e-13) and lie in rcp_mid's
// range.  False if one does not.
template <bool EXACT>
__device__ __forceinline__ bool ldl_solve_t(const double* tot, double lambda, bool fixed_ab, unsigned map,
                                            double* Lm, int lane, double& x)
{
    const unsigned full = 0xffffffffu;
    const int iA = (map >> 12) & 15, kA = (map >> 16) & 15, iB = (map >> 20) & 15, kB = map >> 24;
    const bool dA = iA == kA, dB = iB == kB;                // diagonal entries
    double B = tot[(map >> 6) & 63], A = tot[map & 63];
    B = flip_sign(B, iB == 8);                              // y = -g
    A = flip_sign(A, iA == 8);
    if (fixed_ab) {
        // with (a, b) held fixed their rows and columns become the identity and
        // their right-hand side zero, so the solve gives da = db = 0
        if (iB == 6 || iB == 7) B = 0.0;
        if (kA == 6 || kA == 7 || iA == 6 || iA == 7) A = dA ? 1.0 : 0.0;
    }
    B = fma(dB ? lambda : 0.0, B, B);                       // damped diagonal
    A = fma(dA ? lambda : 0.0, A, A);
    const double a0A = A, a0B = B;
    // the smallest high word of a pivot that passes by its exponent (a damped
    // diagonal that is not positive: none), or any
    const int lo = (1023 - 100) << 20, hi = (1023 + 100) << 20, sl = 42 << 20;
    const int qA = __double2hiint(a0A), qB = __double2hiint(a0B);
    const int loA = !dA ? INT_MIN : qA > 0 ? max(lo, (qA & 0x7ff00000) - sl) : INT_MAX;
    const int loB = !dB ? INT_MIN : qB > 0 ? max(lo, (qB & 0x7ff00000) - sl) : INT_MAX;
    const int hiA = dA ? hi : INT_MAX, hiB = dB ? hi : INT_MAX;
    double rA = 0.0, rB = 0.0, sB = 0.0;                    // 1 / d of the lane's columns
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        const int cj = j == 0 ? 0 : j == 1 ? 8 : ldl_lane(j) - j;   // lane of (i, j) is cj + i
        const double col = j < 2 ? B : A;
        const double piv = __shfl_sync(full, col, cj + j);
        const bool on = kA > j && kA < 8;
        double pB = 0.0;                                    // column 1 first: the next pivot's
        if (j == 0) pB = __shfl_sync(full, col, kB == 1 ? iB : 31) * __shfl_sync(full, col, kB == 1 ? 1 : 31);
        const double pA = __shfl_sync(full, col, on ? cj + iA : 31) * __shfl_sync(full, col, on ? cj + kA : 31);
        const double r = EXACT ? rcp_d(piv) : rcp_mid(piv);
        if (j == 0) B = fma(-pB, r, B);
        A = fma(-pA, r, A);
        if (kB == j) rB = r;
        if (kA == j) rA = r;
        if (j == 2) sB = B * rB;                            // columns 0 and 1 of L, z_0 and z_1
    }
    // L and z = D^-1 y (row 8): every entry times its column's reciprocal;
    // column 7 is the last pivot and z_7 only
    const double piv = __shfl_sync(full, A, 25);
    const double sA = A * rA;
    if (kB < 8) Lm[8 * iB + kB] = sB;
    if (kA < 7) Lm[8 * iA + kA] = sA;
    const double z7 = A * (EXACT ? rcp_d(piv) : rcp_mid(piv));      // lane 26
    bool ok;
    if (EXACT) {
        ok = (!dA || (A > 1e-13 * a0A && A > 0.0)) && (!dB || (B > 1e-13 * a0B && B > 0.0));
    } else {
        const int pA = __double2hiint(A), pB = __double2hiint(B);
        ok = (pA >= loA) & (pA < hiA) & (pB >= loB) & (pB < hiB);
    }
    ok = __all_sync(full, ok);
    __syncwarp();
    // L^T x = z: lane i < 8 holds x_i and its column of L
    double Lcol[8];
#pragma unroll
    for (int j = 1; j < 8; ++j) Lcol[j] = lane < j ? Lm[8 * j + lane] : 0.0;
    x = lane < 7 ? Lm[64 + lane] : 0.0;
    const double x7 = __shfl_sync(full, z7, 26);
    x = fma(-Lcol[7], x7, x);
    if (lane == 7) x = x7;
#pragma unroll
    for (int j = 6; j >= 1; --j) x = fma(-Lcol[j], __shfl_sync(full, x, j), x);
    return ok;
}

// kept out of line: near-singular systems only
static __device__ __noinline__ bool ldl_solve_exact(const double* tot, double lambda, bool fixed_ab, unsigned map,
                                                    double* Lm, int lane, double* x)
{
    return ldl_solve_t<true>(tot, lambda, fixed_ab, map, Lm, lane, *x);
}

// entry (i, k) of the system as doubles (the FP32 elimination's inputs)
__device__ __forceinline__ double ldl_entry(const double* tot, int i, int k, bool fixed_ab)
{
    if (fixed_ab && (k >= 6 || i == 6 || i == 7)) return i == k ? 1.0 : 0.0;
    return i < 8 ? tot[upper_index(k, i)] : -tot[kIdxG + k];
}

// The FP32 elimination of GLT_SOLVE_FP32 (H and g are FP32 sums, relative
// error ~1e-7, so the step they define is known to ~cond x 1e-7 however it is
// solved; the FP32 elimination adds an error of the same order, ~cond x
// 2^-23).  Lanes 0-27 hold the strictly lower entries (i, k), i > k, column by
// column; lanes 0-7 also the diagonal entry and the right-hand side of row
// `lane`.  Used when every FP32 pivot is above 1e-4 of its damped diagonal,
// where its rounding (~1e-6 of the diagonal) cannot change its sign; false
// otherwise: the FP64 elimination decides.
__device__ __forceinline__ bool ldl_solve_warp_fp32(const double* src, double lambda, bool fixed_ab, int lane,
                                                    double& x64)
{
    const unsigned full = 0xffffffffu;
    const int row = lane & 7;
    const int ek = lane < 7 ? 0 : lane < 13 ? 1 : lane < 18 ? 2 : lane < 22 ? 3 : lane < 25 ? 4
                 : lane < 27 ? 5 : lane < 28 ? 6 : 7;
    const int ei = lane < 28 ? lane - (ek * 7 - (ek * (ek - 1)) / 2) + ek + 1 : 8;
    float e = lane < 28 ? f32_of(ldl_entry(src, ei, ek, fixed_ab)) : 0.0f;
    const double diag = ldl_entry(src, row, row, fixed_ab);
    const double a0 = fma(lambda, diag, diag);
    const float a0f = f32_of(a0);
    float dg = a0f, dinv = 0.0f;
    float y = f32_of(ldl_entry(src, 8, row, fixed_ab));
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float d = __shfl_sync(full, dg, j);
        const float r = __frcp_rn(d);
        if (lane == j) dinv = r;
        if (j < 7) {
            const float l = e * r;
            const int cj = j * 7 - (j * (j - 1)) / 2 - j - 1;   // lane of (i, j) is cj + i
            const bool trail = lane < 28 && ek > j;
            const bool drow = lane > j && lane < 8;
            const float li = __shfl_sync(full, l, cj + (trail ? ei : j + 1));
            const float ak = __shfl_sync(full, e, cj + (trail ? ek : j + 1));
            const float ld = __shfl_sync(full, l, cj + (drow ? lane : j + 1));
            const float ad = __shfl_sync(full, e, cj + (drow ? lane : j + 1));
            const float yj = __shfl_sync(full, y, j);
            if (trail) e = fmaf(-li, ak, e);
            if (drow) {
                dg = fmaf(-ld, ad, dg);
                y = fmaf(-ld, yj, y);
            }
            if (lane < 28 && ek == j) e = l;
        }
    }
    if (!__all_sync(full, dg > 1e-4f * a0f || lane >= 8)) return false;
    // column `row` of L (entries below the diagonal) gathered into the row's lane
    float Lcol[8];
#pragma unroll
    for (int i = 1; i < 8; ++i) {
        const int cr = row * 7 - (row * (row - 1)) / 2 - row - 1;
        const float v = __shfl_sync(full, e, row < i ? cr + i : 0);
        Lcol[i] = row < i ? v : 0.0f;
    }
    // diagonal, backward (L^T x = D^-1 y)
    float x = y * dinv;
#pragma unroll
    for (int j = 7; j >= 1; --j) {
        const float xj = __shfl_sync(full, x, j);
        if (row < j) x = fmaf(-Lcol[j], xj, x);
    }
    x64 = f64_of(x);
    return true;
}

// A, B or C (g = 0, 1, 2) beyond theta = 0.01: longer series, or closed forms
static __device__ __noinline__ double se3_coefficient(double th2, int g)
{
    if (th2 < 0.01) {
        const double c4 = g == 0 ? 1.0 / 362880.0 : g == 1 ? 1.0 / 3628800.0 : 1.0 / 39916800.0;
        const double c3 = g == 0 ? -1.0 / 5040.0 : g == 1 ? -1.0 / 40320.0 : -1.0 / 362880.0;
        const double c2 = g == 0 ? 1.0 / 120.0 : g == 1 ? 1.0 / 720.0 : 1.0 / 5040.0;
        const double c1 = g == 0 ? -1.0 / 6.0 : g == 1 ? -1.0 / 24.0 : -1.0 / 120.0;
        const double c0 = g == 0 ? 1.0 : g == 1 ? 0.5 : 1.0 / 6.0;
        return fma(fma(fma(fma(th2, c4, c3), th2, c2), th2, c1), th2, c0);
    }
    const double th = sqrt(th2);
    double sn, cs, sh, ch;
    sincos(th, &sn, &cs);
    sincos(0.5 * th, &sh, &ch);
    return g == 0 ? sn / th : g == 1 ? 2.0 * sh * sh / th2 : (th - sn) / (th2 * th);
}

// exp(delta_xi) of the step xs as a 3x4 [R_e | t_e], entry (r, c) on lane
// 4 r + c:
//   R_e(r, c) = d_rc + A W_rc + B (w_r w_c - d_rc th2)            (W = [w]x)
//   t_e(r)    = v_r + B (w x v)_r + C (w_r (w . v) - v_r th2)
// with A = sin th / th, B = (1 - cos th) / th^2, C = (th - sin th) / th^3.
// Eight FP64 instructions, seven of them on the chain (the one-entry-per-lane
// form with uniform A, B, C took 17 and two compares): three give th2 (lanes
// 0-15), w . v (lane 16) and w x v (lanes 17-19) at once; u = c1 + c2 th2 of
// the series (lanes 12-14) is also -d_rc th2 or -v_r th2 of the entries, and
// u Y + Z the series (Y = th2, Z = c0) and w_r (.) - (.) th2 (Y = 1, Z = w_r
// (.)); two more give the entry.  No select stands between two FP64
// instructions of the chain: a result costs ~50 cycles more on the way out of
// the FP64 pipe than to its next instruction.
__device__ __forceinline__ double se3_exp_warp(const double* xs, unsigned md, unsigned me, int lane)
{
    const unsigned full = 0xffffffffu;
    const double p1 = xs[md & 31], q1 = xs[(md >> 5) & 31], p2 = xs[(md >> 10) & 31], q2 = xs[(md >> 15) & 31],
                 p3 = xs[(md >> 20) & 31], q3 = xs[(md >> 25) & 31];
    const double w = xs[me & 31], wc = xs[(me >> 5) & 31], dd = xs[(me >> 10) & 31], c1 = xs[(me >> 15) & 31];
    const double W = flip_sign(xs[(me >> 20) & 31], (me >> 25) != 0);
    const bool poly = lane >= 12 && lane < 15, rot = (lane & 3) < 3;
    const double s = fma(p3, q3, fma(flip_sign(p2, lane >= 17 && lane < 20), q2, p1 * q1));   // th2 on lanes 0-15
    const double u = fma(-s, dd, c1);
    const double wv = __shfl_sync(full, s, 16);
    const double cr = __shfl_sync(full, s, 17 + (lane >> 2) % 3);
    const double th2 = __shfl_sync(full, s, 0);
    const double Z = w * (rot ? wc : wv);
    double ey = fma(u, poly ? s : 1.0, Z);
    if (!(__double_as_longlong(th2) < 0x3f1a36e2eb1c432dll)) {   // th2 >= 1e-4 (or NaN)
        const double co = se3_coefficient(th2, lane >= 12 ? lane - 12 : 0);
        if (poly) ey = co;
    }
    const double cx = __shfl_sync(full, ey, rot ? 12 : 13);  // of W_rc / (w x v)_r: A / B
    const double cy = __shfl_sync(full, ey, rot ? 13 : 14);  // of ey: B / C
    return fma(cy, ey, fma(cx, rot ? W : cr, dd));
}

// exp(delta_xi) - I in FP32, entry (r, c) on lane 4 r + c (GLT_SOLVE_FP32): its
// entries are O(|delta|), so FP32 rounding leaves ~1e-7 |delta| (absolute).
// Coefficients as above (power series below th^2 = 0.25, truncation < 3e-11
// relative).
__device__ __forceinline__ double se3_exp_minus_i_warp(const double* xs, int lane)
{
    const float v0 = f32_of(xs[0]), v1 = f32_of(xs[1]), v2 = f32_of(xs[2]);
    const float w0 = f32_of(xs[3]), w1 = f32_of(xs[4]), w2 = f32_of(xs[5]);
    const float th2 = fmaf(w0, w0, fmaf(w1, w1, w2 * w2));
    float A, B, Cc;
    if (th2 < 0.25f) {
        A = fmaf(fmaf(fmaf(fmaf(th2, 1.0f / 362880.0f, -1.0f / 5040.0f), th2, 1.0f / 120.0f), th2, -1.0f / 6.0f), th2, 1.0f);
        B = fmaf(fmaf(fmaf(fmaf(th2, 1.0f / 3628800.0f, -1.0f / 40320.0f), th2, 1.0f / 720.0f), th2, -1.0f / 24.0f), th2, 0.5f);
        Cc = fmaf(fmaf(fmaf(fmaf(th2, 1.0f / 39916800.0f, -1.0f / 362880.0f), th2, 1.0f / 5040.0f), th2, -1.0f / 120.0f), th2, 1.0f / 6.0f);
    } else {
        const float th = sqrtf(th2);
        const float sn = sinf(th), sh = sinf(0.5f * th);
        A = sn / th;
        B = 2.0f * sh * sh / th2;
        Cc = (th - sn) / (th2 * th);
    }
    // one element (r, c) of the 3x4 increment per lane 0-11, every lane
    // running the same instructions on its own operands:
    //   (R_e - I)(r, c) = A W_rc + B (w_r w_c - d_rc th2)        (W = [w]x)
    //   t_e(r)          = v_r + B (w x v)_r + C (w_r (w . v) - v_r th2)
    // as  base + cA (a1 b1 - a2 b2) + cB (p q - d th2).
    const float wv = fmaf(w0, v0, fmaf(w1, v1, w2 * v2));
    const int er = (lane >> 2) % 3, ec = lane & 3;
    const float wr = er == 0 ? w0 : (er == 1 ? w1 : w2);
    const float wr1 = er == 0 ? w1 : (er == 1 ? w2 : w0);   // w_{r+1}
    const float wr2 = er == 0 ? w2 : (er == 1 ? w0 : w1);   // w_{r+2}
    const float vr = er == 0 ? v0 : (er == 1 ? v1 : v2);
    const float vr1 = er == 0 ? v1 : (er == 1 ? v2 : v0);
    const float vr2 = er == 0 ? v2 : (er == 1 ? v0 : v1);
    const float wc = ec == 0 ? w0 : (ec == 1 ? w1 : w2);
    const bool rot = ec < 3;
    const float drc = (rot && er == ec) ? 1.0f : 0.0f;
    // W_rc = +w_{r+2} if c = r+1, -w_{r+1} if c = r+2, 0 on the diagonal
    const float Wrc = ec == (er + 1) % 3 ? -wr2 : (ec == (er + 2) % 3 ? wr1 : 0.0f);
    const float base = rot ? 0.0f : vr;
    const float a1 = rot ? Wrc : wr1, b1 = rot ? 1.0f : vr2;
    const float a2 = rot ? 0.0f : wr2, b2 = rot ? 0.0f : vr1;
    const float pq = rot ? wc : wv, dd = rot ? drc : vr;
    const float ex = fmaf(a1, b1, -(a2 * b2));
    const float ey = fmaf(wr, pq, -(dd * th2));
    return f64_of(fmaf(rot ? B : Cc, ey, fmaf(rot ? A : B, ex, base)));
}

// One LM decision after a pass, whose cluster-wide sums are in the buffer
// solver_buffer() named; executed by all 32 lanes of one warp with uniform
// control flow.
// HC: the cached-Hessian form (the sums are g0 = sum w r J_ic, E and n; the
// step is -e^-a H^-1 g0 with the level's per-reference H^-1, since the rows
// are e^a J_ic and the normal matrix e^2a H).
template <bool HC = false>
__device__ inline void solver_step_warp(const StreamDesc& D, Solver& S, PassParams& P, int lane, bool write_trace)
{
    const unsigned full = 0xffffffffu;
    constexpr int kE = HC ? kHcE : kIdxE, kN = HC ? kHcN : kIdxN;
    const int4 w = S.w;
    const unsigned map_ldl = S.map_ldl[lane], map_dot = S.map_dot[lane], map_ent = S.map_ent[lane],
                   map_cmp = S.map_cmp[lane];
    int it = w.x, status = w.y, fl = w.w;
    const int level = fl >> kFlLevel;
    const int wb = (fl & kFlAcc) ? 0 : 1;
    const double* tot = S.tot[wb];
    const int n = S.n[wb];
    const bool sums_finite = S.bad == 0;
    const bool enough = n >= D.min_valid && n > 0 && sums_finite;
    if (!sums_finite) status |= GLT_TRACK_DIVERGED;
    const long long stop_bits = abs_bits(level > 0 ? D.eps_step_coarse : D.eps_step);
    const long long take_bits = abs_bits(D.accept_step);
    double lambda = D.lambda0;
    bool accept = false, load_normal = false, finish = false, candidate = false;
    if (!(fl & kFlCand)) {
        if (!enough) {
            if (sums_finite) status |= GLT_TRACK_TOO_FEW_POINTS;
        } else {
            load_normal = true;
            it = 0;
            candidate = true;
        }
    } else {
        ++it;
        accept = enough && (fl & kFlSmall);
        bool flat = false;
        if (enough && !accept) {
            // c' < c  <=>  E' n < E n' (both sides non-negative: compared through
            // their bits; both products in one instruction);  flat: c' - c <= eps c
            const double* old = S.tot[wb ^ 1];
            const double En = (lane & 1) ? old[kE] * tot[kN] : tot[kE] * old[kN];
            const double e0 = __shfl_sync(full, En, 0), e1 = __shfl_sync(full, En, 1);
            accept = __double_as_longlong(e0) < __double_as_longlong(e1);
            if (!accept && __double_as_longlong(D.eps_cost) != 0) flat = e0 - e1 <= D.eps_cost * e1;
        }
        lambda = S.lam[accept ? 0 : 1];
        load_normal = accept;
        if (accept) fl = (fl ^ kFlCur) | kFlMoved;
        if (it >= D.max_iters[level] || (fl & kFlStop) || flat)
            finish = true;
        else
            candidate = true;
    }
    // the normal equations of the accepted state: this pass's, or the kept
    // ones after a rejection
    if (load_normal) fl ^= kFlAcc;
    const double* src = S.tot[(fl & kFlAcc) ? 1 : 0];
    bool solved = false;
    double x = 0.0;                  // delta, entry i on lane i < 8
    if (HC && candidate && !(w.w & kFlCand)) {
        // -e^-a H^-1 of the level, kept for its later passes
        const double* Hi = D.Hc + 72 * level + 36;
        const double h0 = Hi[lane], h1 = Hi[lane < 4 ? 32 + lane : 0];
        S.Hi[lane] = -S.ema * h0;
        if (lane < 4) S.Hi[32 + lane] = -S.ema * h1;
        if (lane == 0) S.hc_ok = abs_bits(h0) < kInfBits;
        __syncwarp();
    }
    if (candidate && HC) {
        // ---- delta = -e^-a H^-1 g0, half a row per lane (rows 0-5 on lanes 0-5
        // and 8-13); the affine pair is held fixed in this form
        if (S.hc_ok) {
            const int r6 = (lane & 7) < 6 ? (lane & 7) : 0, c0 = (lane & 8) ? 3 : 0;
            const double* h = S.Hi + 6 * r6 + c0;
            x = fma(h[0], src[c0], fma(h[1], src[c0 + 1], h[2] * src[c0 + 2]));
            x += __shfl_xor_sync(full, x, 8);
            if (lane == 6 || lane == 7) x = 0.0;
            solved = true;
        }
    } else if (candidate) {
        if (D.solve != GLT_SOLVE_FP64) solved = ldl_solve_warp_fp32(src, lambda, !D.affine, lane, x);
        if (!solved) {
            solved = ldl_solve_t<false>(src, lambda, !D.affine, map_ldl, S.Lm, lane, x);
            if (!solved) {
                double xe = 0.0;
                solved = ldl_solve_exact(src, lambda, !D.affine, map_ldl, S.Lm, lane, &xe);
                x = xe;
            }
        }
    }
    if (candidate && !solved) {
        status |= GLT_TRACK_NOT_PD;
        finish = true;
    }
    bool evaluated = false;          // P already holds the next state
    if (solved) {
        const bool fp32 = D.solve == GLT_SOLVE_FP32;
        if (lane < 8) S.xs[lane] = x;
        __syncwarp();
        // ---- Tc = T exp(delta) (FP32 form: T + T (exp(delta) - I)), three FP64
        // instructions on all lanes: entry (r, c) on lane 16 + 4 r + c, the same
        // minus the identity (what the pass parameters need) on lane 4 r + c,
        // a + da and b + db on lanes 12 and 13, the two next dampings on 14, 15
        const double ent = fp32 ? se3_exp_minus_i_warp(S.xs, lane) : se3_exp_warp(S.xs, map_dot, map_ent, lane);
        const double* T = S.st[fl & kFlCur];
        const double t0 = T[map_cmp & 31], t1 = T[(map_cmp >> 5) & 31], t2 = T[(map_cmp >> 10) & 31];
        double add = T[(map_cmp >> 15) & 31];
        const int q = lane & 15, ec = q & 3;
        if (fp32 && q < 12) {
            add = T[q];
            if (lane == 0 || lane == 5 || lane == 10)
                asm volatile("add.rn.f64 %0, %0, 0dBFF0000000000000;" : "+d"(add));   // never speculated
        }
        const double xab = S.xs[6 + (lane & 1)];
        const double x0 = __shfl_sync(full, ent, ec), x1 = __shfl_sync(full, ent, 4 + ec),
                     x2 = __shfl_sync(full, ent, 8 + ec);
        const double v = fma(t0, x0, fma(t1, x1, fma(t2, q < 12 ? x2 : lane < 14 ? xab : lambda, add)));
        // (t0 = t1 = 0 on lanes 12-15 and 28-31 drop x0, x1 unless those are not
        // finite, which lanes 0-11 report as well)
        // a step below the level's stop threshold (and below accept_step)
        // would be taken whatever its cost and would end the level, so it
        // is taken here without a pass of its own: the next level's start
        // pass is the first evaluation of the new state; on the finest
        // level the result keeps the cost and count of the last evaluated
        // state
        const long long xb = abs_bits(x);
        const bool small = __all_sync(full, xb < take_bits || lane >= 6);
        const bool stop = __all_sync(full, xb < stop_bits || lane >= 6);
        if (!__all_sync(full, abs_bits(v) < kInfBits || lane == 14 || lane == 15 || lane >= 28)) {
            // the solve produced a state that is not finite: keep the
            // accepted one and end the level
            status |= GLT_TRACK_DIVERGED;
            finish = true;
        } else {
            // the next pass evaluates the new state either way
            const float vf = f32_rn(v);
            const float ea = expf(vf);
            const int nx = (fl & kFlCur) ^ 1;
            if (lane < 14) reinterpret_cast<float*>(&P)[map_cmp >> 20] = lane == 12 ? ea : vf;
            double* pd = lane < 14 ? &S.st[nx][lane] : lane < 16 ? &S.lam[lane - 14] : &S.st[nx][lane - 16];
            if (lane >= 12 && lane < 28) *pd = v;
            evaluated = true;
            fl = (fl & ~(kFlSmall | kFlStop)) | kFlCand | (small ? kFlSmall : 0) | (stop ? kFlStop : 0);
            if (small && stop) {
                ++it;
                finish = true;
                fl = (fl ^ kFlCur) | kFlMoved;
            }
        }
    }
    // commit the pass outcome
    if (write_trace && lane == 0 && D.trace_E && w.z < D.max_trace) {
        D.trace_E[w.z] = tot[kE];
        D.trace_n[w.z] = n;
        D.trace_info[w.z] = level * 4 + ((w.w & kFlCand) ? 1 + (accept ? 2 : 0) : 0);
    }
    if (finish && lane == 0) {
        S.iters[level] = it;
        S.res_E = src[kE];
        S.res_n = S.n[(fl & kFlAcc) ? 1 : 0];
    }
    if (!candidate || finish) {
        // the next level, from the accepted state
        int l = level;
        do --l;
        while (l >= 0 && D.max_iters[l] <= 0);
        double* T = S.st[fl & kFlCur];
        __syncwarp();
        if (l < 0) {
            // GLT_SOLVE_FP32: the poses composed from FP32 increments drift
            // from orthonormal by ~1e-9 per step: one Newton step R' = R (3 I - R^T R) / 2 =
            // R + R (I - R^T R) / 2 on the final pose (FP64; the deviation
            // becomes its square)
            if ((fl & kFlMoved) && D.solve == GLT_SOLVE_FP32) {
                const int i = lane / 3, j = lane % 3;
                double dlt = lane < 9 ? (i == j ? 1.0 : 0.0) : 0.0;
                if (lane < 9) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) dlt = fma(-T[4 * k + i], T[4 * k + j], dlt);
                }
                const int r = lane >> 2, c = lane & 3;
                const int cc = c < 3 ? c : 0;
                const double d0 = __shfl_sync(full, dlt, cc), d1 = __shfl_sync(full, dlt, 3 + cc),
                             d2 = __shfl_sync(full, dlt, 6 + cc);
                double v = 0.0;
                if (lane < 12 && c < 3)
                    v = fma(0.5, fma(T[4 * r], d0, fma(T[4 * r + 1], d1, T[4 * r + 2] * d2)), T[lane]);
                __syncwarp();
                if (lane < 12 && c < 3) T[lane] = v;
            }
            if (lane == 0) P.done = 1;
        } else {
            fl = (fl & ((1 << kFlLevel) - 1) & ~kFlCand) | (l << kFlLevel);
            if (!evaluated)
                make_pass_params_warp(T, T[12], T[13], l, P, lane);
            else if (lane == 13) {
                P.level = l;
                P.scale = ldexpf(1.0f, -l);
            }
        }
    }
    if (lane == 0) {
        S.w = make_int4(it, status, w.z + 1, fl);
        S.bad = 0;
    }
    __syncwarp();
}

__device__ inline void solver_write_result(const StreamDesc& D, const Solver& S, glt_result* out)
{
    const double* T = S.st[S.w.w & kFlCur];
    if (D.trace_count) *D.trace_count = S.w.z;
    for (int i = 0; i < 12; ++i) out->T[i] = T[i];
    out->a = T[12];
    out->b = T[13];
    out->cost = S.res_n > 0 ? S.res_E / (double)S.res_n : S.res_E;
    out->n_valid = S.res_n;
    int tot = 0;
    for (int l = 0; l < kMaxLevels; ++l) {
        out->iters[l] = S.iters[l];
        tot += S.iters[l];
    }
    out->iters_total = tot;
    out->passes = S.w.z;
    out->status = S.w.y;
}

}  // namespace glt
