// Map-point upload (GLidE-SLAM Sec. IV-C "Precompute"): back-project each
// point and sample its reference patch I0 at the pattern offsets on every
// REF level (Eq. 2's I0(u_i^0 + du_k)); in the inverse-compositional form
// also the reference gradient there (the image part of the cached Jacobian
// rows of Sec. IV-B; the geometric part at x_r follows from the point).
#include <algorithm>

#include "glt_internal.h"

namespace glt {

// A level-l reference position u0 / 2^l is exact in FP32; a point's samples
// share its fractional part, so their bilinear weights are computed once.  A
// point is unusable on a level (its first sample is NaN) if its depth is not
// positive or a sample leaves 1 <= q < W-2, 1 <= q < H-2.
struct RefLevels {
    const uint8_t* img[kMaxLevels];
#ifdef GLT_CHECKED
    size_t size[kMaxLevels];     // bytes of a level
    __device__ __forceinline__ size_t bytes(int l) const { return size[l]; }
#else
    __device__ __forceinline__ size_t bytes(int) const { return 0; }
#endif
};

struct RefPoint {
    int xb, yb;
    float w00, w10, w01, w11;
    bool ok;
};

__device__ __forceinline__ RefPoint ref_point(const LevelDev& lv, float u0, float v0, float d, int l, int h)
{
    RefPoint r;
    const bool finite = isfinite(u0) && isfinite(v0) && isfinite(d) && d > 0.0f &&
                        fabsf(u0) < 1e7f && fabsf(v0) < 1e7f;
    const float s = ldexpf(1.0f, -l);
    const float U = u0 * s, V = v0 * s;
    const float fu = floorf(U), fv = floorf(V);
    r.xb = finite ? (int)fu : -1000;
    r.yb = finite ? (int)fv : -1000;
    // every sample q = (U + dx, V + dy) must satisfy 1 <= q < W-2, 1 <= q < H-2
    r.ok = finite && r.xb >= 1 + h && r.xb <= lv.W - 3 - h && r.yb >= 1 + h && r.yb <= lv.H - 3 - h;
    const float al = U - fu, be = V - fv;
    r.w00 = (1.0f - al) * (1.0f - be);
    r.w10 = al * (1.0f - be);
    r.w01 = (1.0f - al) * be;
    r.w11 = al * be;
    return r;
}

// p, from where n words of the level (img, size bytes) are read
template <class T>
__device__ __forceinline__ const T* level_read(const uint8_t* img, size_t size, const uint8_t* p, size_t n)
{
    return checked(reinterpret_cast<const T*>(p), n, reinterpret_cast<const T*>(img), size / sizeof(T), CK_IMAGE);
}

// tab + i, where n elements are written; null without a table
template <class T>
__device__ __forceinline__ T* table_to(const StreamDesc& D, T* tab, size_t i, size_t n)
{
    return tab ? checked(tab + i, n, tab, table_size(D.L, D.Npad, D.pattern, D.tg), CK_SET_POINTS) : nullptr;
}

// The 8-pixel pattern of one point on one level.
__device__ __forceinline__ void set_pattern8(const StreamDesc& D, const RefPoint& r, const uint8_t* img, size_t size, int P, int l, int p,
                                             float* I0, float2* G0)
{
    // the samples' and gradients' taps: 8 x 8 bytes from (xb - 3, yb - 3)
    const uint8_t* win = nullptr;
    if (r.ok) win = level_read<uint8_t>(img, size, img + (size_t)(r.yb - 3) * P + (r.xb - 3), (size_t)7 * P + 8);
    I0 = table_to(D, I0, ((size_t)l * D.Npad + p) * 8, 8);
    G0 = table_to(D, G0, ((size_t)l * D.Npad + p) * 8, 8);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (!r.ok) {
            I0[k] = k == 0 ? __int_as_float(0x7fc00000) : 0.0f;
            if (G0) G0[k] = make_float2(0.0f, 0.0f);
            continue;
        }
        const uint8_t* t = win + (3 + pat_dy(k)) * P + (3 + pat_dx(k));
        const float I00 = t[0], I10 = t[1], I01 = t[P], I11 = t[P + 1];
        I0[k] = fmaf(r.w00, I00, fmaf(r.w10, I10, fmaf(r.w01, I01, r.w11 * I11)));
        if (G0) {
            // central differences at the four taps, bilinear weights, then the 1/2
            const float gx = 0.5f * fmaf(r.w00, I10 - (float)t[-1],
                                    fmaf(r.w10, (float)t[2] - I00,
                                    fmaf(r.w01, I11 - (float)t[P - 1], r.w11 * ((float)t[P + 2] - I01))));
            const float gy = 0.5f * fmaf(r.w00, I01 - (float)t[-P],
                                    fmaf(r.w10, I11 - (float)t[1 - P],
                                    fmaf(r.w01, (float)t[2 * P] - I00, r.w11 * ((float)t[2 * P + 1] - I10))));
            G0[k] = make_float2(gx, gy);
        }
    }
}

// Group g (of TG) of rows of the PS x PS patch of one point on one level: the
// group's window, one row and column beyond it on each side and one more below
// and to the right, is read once with aligned 8-byte loads (those that hold a
// byte of it) and every sample and gradient is interpolated from registers.
template <int PS, int TG>
__device__ __forceinline__ void set_patch(const StreamDesc& D, const RefPoint& r, const uint8_t* img, size_t size, int P, int l, int p,
                                          int g, float* I0, float2* G0)
{
    constexpr int h = (PS - 1) / 2, RG = group_rows(PS, TG), R = RG + 3, NB = PS + 3, NW = (NB + 3) / 4;
    const int j0 = g * RG, rows = min(RG, PS - j0);
    const size_t stride = (size_t)D.Npad * TG, at0 = ((size_t)l * group_samples(PS, TG)) * stride + (size_t)p * TG + g;
    I0 = table_to(D, I0, at0, (size_t)(rows * PS - 1) * stride + 1);
    G0 = table_to(D, G0, at0, (size_t)(rows * PS - 1) * stride + 1);
    if (!r.ok) {
#pragma unroll
        for (int q = 0; q < RG * PS; ++q) {
            if (q >= rows * PS) break;
            I0[q * stride] = q == 0 && g == 0 ? __int_as_float(0x7fc00000) : 0.0f;
            if (G0) G0[q * stride] = make_float2(0.0f, 0.0f);
        }
        return;
    }
    const int xs = r.xb - h - 1, ys = r.yb - h - 1 + j0, a8 = xs & ~7, sh = xs - a8;
    const bool wide = sh + NB > 16, far = sh >= 4;
    uint32_t win[R][NW];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        if (q < rows + 3) {
            const uint2* rp = level_read<uint2>(img, size, img + (size_t)(ys + q) * P + a8, wide ? 3 : sh + NB > 8 ? 2 : 1);
            const uint2 u0 = rp[0], u1 = (sh + NB > 8) ? rp[1] : make_uint2(0u, 0u), u2 = wide ? rp[2] : make_uint2(0u, 0u);
            const uint32_t v[7] = {u0.x, u0.y, u1.x, u1.y, u2.x, u2.y, 0u};
#pragma unroll
            for (int i = 0; i < NW; ++i)
                win[q][i] = __funnelshift_r(far ? v[i + 1] : v[i], far ? v[i + 2] : v[i + 1], 8 * sh);   // (modulo 32)
        } else {
#pragma unroll
            for (int i = 0; i < NW; ++i) win[q][i] = 0u;
        }
    }
    auto px = [&](int y, int x) { return u8f(win[y][x >> 2], x & 3); };   // window row y, column x (sample (0, 0) at (1, 1))
#pragma unroll
    for (int j = 0; j < RG; ++j) {
        if (j >= rows) break;
#pragma unroll
        for (int i = 0; i < PS; ++i) {
            const int y = j + 1, x = i + 1;
            const size_t at = (j * PS + i) * stride;
            const float I00 = px(y, x), I10 = px(y, x + 1), I01 = px(y + 1, x), I11 = px(y + 1, x + 1);
            I0[at] = fmaf(r.w00, I00, fmaf(r.w10, I10, fmaf(r.w01, I01, r.w11 * I11)));
            if (G0) {
                const float gx = 0.5f * fmaf(r.w00, I10 - px(y, x - 1),
                                        fmaf(r.w10, px(y, x + 2) - I00,
                                        fmaf(r.w01, I11 - px(y + 1, x - 1), r.w11 * (px(y + 1, x + 2) - I01))));
                const float gy = 0.5f * fmaf(r.w00, I01 - px(y - 1, x),
                                        fmaf(r.w10, I11 - px(y - 1, x + 1),
                                        fmaf(r.w01, px(y + 2, x) - I00, r.w11 * (px(y + 2, x + 1) - I10))));
                G0[at] = make_float2(gx, gy);
            }
        }
    }
}

// One thread per (point, group) and level (grid.y).  One thread per point over
// all levels and samples, with byte loads, left the chip empty.  2000 points,
// 11 x 11 patches, 6 levels: 12 us; with the two kernels below the whole refresh
// of a reference went from 520 to 70 us.
__global__ void __launch_bounds__(128)
set_points_kernel(StreamDesc* __restrict__ desc, int n, RefLevels ref, const float* __restrict__ uvd, float cx, float cy,
                  float4* __restrict__ pt, float2* __restrict__ dz, float* __restrict__ I0, float2* __restrict__ G0)
{
    const StreamDesc& D = *desc;
    const int t = blockIdx.x * blockDim.x + threadIdx.x, l = blockIdx.y;
    if (t == 0 && l == 0) desc->N = n;      // the point count the kernels of later passes read
    const int tg = D.tg, p = t / tg, g = t - p * tg;
    if (p >= n) return;
    const float u0 = uvd[3 * p], v0 = uvd[3 * p + 1], d = uvd[3 * p + 2];
    if (l == 0 && g == 0) {
        *checked(pt + p, 1, pt, (size_t)D.Npad, CK_SET_POINTS) = make_float4(u0, v0, (u0 - cx) / D.fx, (v0 - cy) / D.fy);
        *checked(dz + p, 1, dz, (size_t)D.Npad, CK_SET_POINTS) = make_float2(d, 1.0f / d);
    }
    const LevelDev& lv = D.lv[l];
    const RefPoint r = ref_point(lv, u0, v0, d, l, D.pattern ? (D.pattern - 1) / 2 : 2);
    const uint8_t* img = ref.img[l];
    const size_t size = ref.bytes(l);
    switch (D.pattern * 8 + tg) {
    case 1: set_pattern8(D, r, img, size, lv.pitch, l, p, I0, G0); break;
    case 3 * 8 + 1: set_patch<3, 1>(D, r, img, size, lv.pitch, l, p, g, I0, G0); break;
    case 5 * 8 + 1: set_patch<5, 1>(D, r, img, size, lv.pitch, l, p, g, I0, G0); break;
    case 7 * 8 + 1: set_patch<7, 1>(D, r, img, size, lv.pitch, l, p, g, I0, G0); break;
    case 9 * 8 + 1: set_patch<9, 1>(D, r, img, size, lv.pitch, l, p, g, I0, G0); break;
    case 11 * 8 + 1: set_patch<11, 1>(D, r, img, size, lv.pitch, l, p, g, I0, G0); break;
    case 7 * 8 + kHcGroups: set_patch<7, kHcGroups>(D, r, img, size, lv.pitch, l, p, g, I0, G0); break;
    case 11 * 8 + kHcGroups: set_patch<11, kHcGroups>(D, r, img, size, lv.pitch, l, p, g, I0, G0); break;
    }
}

// Sec. IV-B: with the inverse-compositional rows J_ik evaluated on the
// reference, H = sum_i sum_k J_ik^T J_ik is fixed while the reference is;
// Sec. IV-C "Precompute IC": each point's H_i is reduced into one H per level.
// Two kernels:
//  * hess_points_kernel: a thread sums the 21 upper-triangle products of one
//    point's rows on one level in FP32 (J_k = [Jt_k, x_r x Jt_k], Jt_k = gx_k a0
//    + gy_k a1 with the cached reference gradient and the projection rows at
//    x_r, e^a = 1);
//  * hess_finish_kernel: one block per sum and level adds the points in FP64
//    (256 interleaved chains, then a tree), so that the FP64 pipes of many SMs
//    share the additions; the level's last block factorises H = L D L^T on one
//    warp, row i on lane i (pivots d > 0 and d > 1e-13 H_jj, else H^-1[0] = NaN:
//    not positive definite), and solves for column c of H^-1 on lane c.
// A point's samples and a chain's points stay in order, so that the sums and the
// factors are those of one block per level with a serial factorisation, bit for
// bit; that took 118 (7 x 7) to 192 us (11 x 11) for 2000 points, these 26 + 18.
// Bound by the chains: 121 samples of a point, 8 points, 6 columns.
constexpr int kHessThreads = 128, kHessChains = 256;

__global__ void __launch_bounds__(kHessThreads)
hess_points_kernel(const StreamDesc* __restrict__ desc, float* __restrict__ part)
{
    const StreamDesc& D = *desc;
    const int l = blockIdx.y, p = blockIdx.x * kHessThreads + threadIdx.x;
    if (p >= D.N) return;
    const float s = ldexpf(1.0f, -l);
    const int tg = D.tg, ps = D.pattern, RG = ps ? group_rows(ps, tg) : 0, SG = ps ? group_samples(ps, tg) : 0;
    const size_t stride = ps ? (size_t)D.Npad * tg : 1;
    const size_t base = ps ? ((size_t)l * SG * D.Npad + p) * tg : ((size_t)l * D.Npad + p) * 8;
    float h[kHessSums];
#pragma unroll
    for (int i = 0; i < kHessSums; ++i) h[i] = 0.0f;
    float* out = checked(part + (size_t)l * kHessSums * D.Npad + p, (size_t)(kHessSums - 1) * D.Npad + 1, part,
                         (size_t)D.L * kHessSums * D.Npad, CK_TABLE);
    // a point that is not usable on this level of the reference adds zeros
    const bool usable = !isnan(*table_from(D, D.I0, base, 1));
    const float4 q = *checked(D.pt + p, 1, D.pt, (size_t)D.Npad, CK_POINTS);
    const float2 dz = *checked(D.dz + p, 1, D.dz, (size_t)D.Npad, CK_POINTS);
    const float fxl = D.fx * s * dz.y, fyl = D.fy * s * dz.y;
    const float a0[3] = {fxl, 0.0f, -fxl * q.z};
    const float a1[3] = {0.0f, fyl, -fyl * q.w};
    const float xr[3] = {dz.x * q.z, dz.x * q.w, dz.x};
    // the samples in order, a group's (or the pattern's) at a time
    const int groups = !usable ? 0 : ps ? tg : 1;
    for (int g = 0; g < groups; ++g) {
        const int m = ps ? min(RG, ps - g * RG) * ps : 8;
        const float2* G = table_from(D, D.G0, base + g, (size_t)(m - 1) * stride + 1);
#pragma unroll 4
        for (int k = 0; k < m; ++k) {
            const float2 g0 = G[k * stride];
            float J[6];
            J[0] = fmaf(g0.x, a0[0], g0.y * a1[0]);
            J[1] = fmaf(g0.x, a0[1], g0.y * a1[1]);
            J[2] = fmaf(g0.x, a0[2], g0.y * a1[2]);
            J[3] = fmaf(xr[1], J[2], -xr[2] * J[1]);
            J[4] = fmaf(xr[2], J[0], -xr[0] * J[2]);
            J[5] = fmaf(xr[0], J[1], -xr[1] * J[0]);
            int idx = 0;
#pragma unroll
            for (int i = 0; i < 6; ++i)
#pragma unroll
                for (int j = i; j < 6; ++j) {
                    h[idx] = fmaf(J[i], J[j], h[idx]);
                    ++idx;
                }
        }
    }
#pragma unroll
    for (int i = 0; i < kHessSums; ++i) out[(size_t)i * D.Npad] = h[i];
}

__global__ void __launch_bounds__(kHessChains)
hess_finish_kernel(const StreamDesc* __restrict__ desc, const float* __restrict__ part, unsigned* __restrict__ count,
                   double* __restrict__ Hc)
{
    __shared__ double red[kHessChains];
    __shared__ double Ls[6][6], ds[6];
    __shared__ int last;
    const StreamDesc& D = *desc;
    const int e = blockIdx.x, l = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    const float* in = checked(part + ((size_t)l * kHessSums + e) * D.Npad, (size_t)D.N, part, (size_t)D.L * kHessSums * D.Npad, CK_TABLE);
    double acc = 0.0;
#pragma unroll 4
    for (int p = tid; p < D.N; p += kHessChains) acc += (double)in[p];
    red[tid] = acc;
    __syncthreads();
    for (int half = kHessChains / 2; half > 0; half >>= 1) {
        if (tid < half) red[tid] += red[tid + half];
        __syncthreads();
    }
    double* out = Hc + 72 * l;
    if (tid == 0) {
        int i = 0, off = e;                       // (i, j) of upper-triangle entry e
        while (off >= 6 - i) off -= 6 - i++;
        out[6 * i + i + off] = red[0];
        out[6 * (i + off) + i] = red[0];
        __threadfence();
        last = atomicAdd(count + l, 1u) == (unsigned)kHessSums - 1u;
    }
    __syncthreads();
    if (!last || tid >= 32) return;
    __threadfence();
    if (lane == 0) count[l] = 0u;                 // ready for the next reference
    // column by column: d_j and the column of L below it, row i on lane i
    const int r = lane < 6 ? lane : 5;
    double a[6], L[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        a[j] = __ldcg(out + 6 * r + j);
        L[j] = 0.0;
    }
    bool pd = true;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double v = a[j];
#pragma unroll
        for (int k = 0; k < j; ++k) v = fma(-__dmul_rn(L[k], Ls[j][k]), ds[k], v);
        const double dj = __shfl_sync(0xffffffffu, v, j), hj = __shfl_sync(0xffffffffu, a[j], j);
        pd = pd && dj > 0.0 && dj > 1e-13 * hj;
        L[j] = lane == j ? 1.0 : v / dj;
        if (lane < 6 && lane > j) Ls[lane][j] = L[j];
        if (lane == j) ds[j] = dj;
        __syncwarp();
    }
    // column `lane` of H^-1: L y = e, z = D^-1 y, L^T x = z
    double x[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        double y = i == r ? 1.0 : 0.0;
#pragma unroll
        for (int k = 0; k < i; ++k) y = fma(-Ls[i][k], x[k], y);
        x[i] = y;
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        double v = x[i] / ds[i];
#pragma unroll
        for (int k = i + 1; k < 6; ++k) v = fma(-Ls[k][i], x[k], v);
        x[i] = v;
    }
    if (lane < 6) {
#pragma unroll
        for (int i = 0; i < 6; ++i) out[36 + 6 * i + lane] = pd ? x[i] : __longlong_as_double(0x7ff8000000000000ll);
    }
}

cudaError_t launch_ic_hessian(const glt_tracker* t, cudaStream_t s)
{
    if (t->N > 0)
        hess_points_kernel<<<dim3((unsigned)((t->N + kHessThreads - 1) / kHessThreads), (unsigned)t->L), kHessThreads, 0, s>>>(
            t->desc_dev, t->Hpart);
    hess_finish_kernel<<<dim3(kHessSums, (unsigned)t->L), kHessChains, 0, s>>>(t->desc_dev, t->Hpart, t->Hcount, t->Hc);
    return cudaGetLastError();
}

cudaError_t launch_set_points(const glt_tracker* t, const float* uvd_dev, int n, cudaStream_t s)
{
    const int threads = 128;
    const long long tasks = (long long)n * t->desc_host.tg;
    const long long blocks = tasks > 0 ? (tasks + threads - 1) / threads : 1;
    RefLevels ref{};
    for (int l = 0; l < t->L; ++l) {
        ref.img[l] = t->pyr[GLT_REF].base + t->pyr[GLT_REF].off[l];
#ifdef GLT_CHECKED
        ref.size[l] = (size_t)t->pitch[l] * t->H[l];
#endif
    }
    set_points_kernel<<<dim3((unsigned)blocks, (unsigned)t->L), threads, 0, s>>>(
        t->desc_dev, n, ref, uvd_dev, (float)t->cfg.cx, (float)t->cfg.cy, t->pt, t->dz, t->I0, t->G0);
    return cudaGetLastError();
}

#ifdef GLT_CHECKED
unsigned check_flags_points()
{
    unsigned v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_check_flags, sizeof(v));
    cudaMemcpyToSymbol(g_check_flags, &z, sizeof(z));
    return v;
}

// Positive control of the map-point kernels: descriptions that claim less than
// the buffers hold (a level of 8 rows instead of 48, arrays of 32 points instead
// of 64), so that the checks send accesses back that would have been in range.
// *caught: every kernel set the flags of what it accesses.
cudaError_t probe_points(bool* caught)
{
    constexpr int W = 64, H = 48, P = 80, N = 64, CLAIM = 32;
    constexpr size_t TAB = (size_t)128 * N * kHcGroups;      // any pattern's table
    struct Buffers {
        StreamDesc desc;
        alignas(16) uint8_t img[P * H];
        float uvd[3 * N];
        alignas(16) float4 pt[N];
        float2 dz[N];
        alignas(16) float I0[TAB];
        alignas(16) float2 G0[TAB];
        float part[kHessSums * N];
        double Hc[72];
        unsigned count;
    };
    Buffers* B = nullptr;
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&B), sizeof(Buffers));
    if (e != cudaSuccess) return e;
    auto flags = [&](unsigned want) {
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return false;
        return (check_flags_points() & want) == want;
    };
    *caught = true;
    for (const int pattern : {0, 5, 7}) {
        StreamDesc D{};
        D.L = 1;
        D.N = N;
        D.Npad = CLAIM;
        D.fx = D.fy = 50.0f;
        D.pattern = pattern;
        D.K = pattern ? pattern * pattern : 8;
        D.tg = hc_groups(pattern);
        D.lv[0].W = W;
        D.lv[0].H = H;
        D.lv[0].pitch = P;
        D.pt = B->pt;
        D.dz = B->dz;
        D.I0 = B->I0;
        D.G0 = B->G0;
        float uvd[3 * N];
        for (int i = 0; i < N; ++i) {
            uvd[3 * i] = 16.0f + i % 32;
            uvd[3 * i + 1] = 20.0f + i % 8;
            uvd[3 * i + 2] = 2.0f;
        }
        if (e == cudaSuccess) e = cudaMemset(B, 0, sizeof(Buffers));
        if (e == cudaSuccess) e = cudaMemcpy(&B->desc, &D, sizeof(D), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(B->uvd, uvd, sizeof(uvd), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) break;
        RefLevels ref{};
        ref.img[0] = B->img;
        ref.size[0] = (size_t)P * 8;
        set_points_kernel<<<(N * D.tg + 127) / 128, 128>>>(&B->desc, N, ref, B->uvd, 32.0f, 24.0f, B->pt, B->dz, B->I0, B->G0);
        *caught = flags((1u << CK_IMAGE) | (1u << CK_SET_POINTS)) && *caught;
        hess_points_kernel<<<1, kHessThreads>>>(&B->desc, B->part);
        *caught = flags((1u << CK_TABLE) | (1u << CK_POINTS)) && *caught;
        hess_finish_kernel<<<kHessSums, kHessChains>>>(&B->desc, B->part, &B->count, B->Hc);
        *caught = flags(1u << CK_TABLE) && *caught;
    }
    cudaFree(B);
    return e;
}
#endif

}  // namespace glt
