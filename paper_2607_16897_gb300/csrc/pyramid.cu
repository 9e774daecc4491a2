// Image pyramid kernels (GLidE-SLAM Sec. IV-C "Image pyramids": blur, then
// downsample; level 0 is the full-resolution frame).
//
// Level l from level l-1: out(x, y) = (sum_{i,j=-2..2} w_i w_j in(2x+i, 2y+j) + 128) >> 8
// with w = [1 4 6 4 1], clamp-to-edge, computed exactly in integers.  A thread
// makes 8 x 4 outputs in registers: it reads the 16 columns and 11 rows above
// them with 16-byte loads, all issued before the first use, takes the three
// columns beyond from its neighbours' registers, filters each row horizontally
// (two outputs per 32-bit lane pair) and then five rows vertically.  The blocks
// of a level are cut from the flat list of its threads, a whole batch of streams
// in one launch.  Level 1 reads the caller's frame and writes the level-0 copy
// from its registers, so a frame is read from HBM once.
#include <algorithm>

#include "glt_internal.h"

namespace glt {

namespace {
constexpr int PX = 8, PY = 4;        // outputs of a thread
constexpr int PR = 2 * PY + 3;       // input rows of a thread
constexpr int PYR_THREADS = 128;
}  // namespace

// Blocks of a level of dW x dH outputs.
__host__ __device__ int pyr_blocks(int dW, int dH)
{
    return (((dW + PX - 1) / PX) * ((dH + PY - 1) / PY) + PYR_THREADS - 1) / PYR_THREADS;
}

// One block of a launch: the level job (for level 1 with the caller's frame as
// its source and the level-0 buffer as copy0) and its place in the job.
struct Tile {
    PyrJob J;
    uint8_t* copy0;
    int cp, local;
};

// Block f of the launch: tile_map[f] = (job << 16) | block within the job, or,
// for one job without a map, f itself.
__device__ __forceinline__ Tile tile_at(const PyrJob* __restrict__ jobs, const unsigned* __restrict__ tile_map,
                                        const uint8_t* const* frames, const uint8_t* src, int sp, int f)
{
    int z = 0;
    Tile t;
    t.local = f;
    if (tile_map) {
        const unsigned m = tile_map[f];
        z = (int)(m >> 16);
        t.local = (int)(m & 0xffffu);
    }
    t.J = jobs[z];
    t.copy0 = nullptr;
    t.cp = 0;
    if (frames || src) {
        // level 1 from the caller's frame; the blocks also write the level-0 copy
        t.copy0 = const_cast<uint8_t*>(t.J.src);
        t.cp = t.J.sp;
        t.J.src = frames ? frames[z] : src;
        t.J.sp = frames ? t.J.sW : sp;
    }
    return t;
}

// Source loads are L2 loads: a level written by the previous kernel of a
// programmatic chain, or a frame of which nothing is read twice but the rows
// that two threads share.
template <class T>
__device__ __forceinline__ T src_load(const PyrJob& J, const uint8_t* p)
{
    return __ldcg(reinterpret_cast<const T*>(checked(p, sizeof(T), J.src, (size_t)J.sp * J.sH, CK_PYR_SRC)));
}
__device__ __forceinline__ uint32_t src_byte(const PyrJob& J, const uint8_t* row, int x)
{
    return src_load<uint8_t>(J, row + min(max(x, 0), J.sW - 1));
}

// One level of S streams, PX x PY outputs a thread.  For level 1 the source can
// be the caller's frame instead of the level-0 buffer: `frames` (a device table
// of S contiguous frames, pitch = width) or `src` / `sp` (one stream); the
// threads then also write the level-0 copy into the job's source buffer.
//
// Bound in a batch by the loads in flight (256 frames of 640 x 480, 4 levels:
// 62 us, 43% of the copy bandwidth), for one frame by the launch and one memory
// round trip.  8 x 4 outputs: 16-byte loads, three rows in eleven read twice
// (from L2), 44 words a thread in flight, ~16 instructions an output; five blocks
// an SM cost 48 bytes of spills.  Staging 64 x 16 tiles in shared memory with
// 4-byte loads was bound by issue (~150 instructions an output): 136 us for the
// batch, 47 instead of 23 us for 64 frames of mixed sizes.
__global__ void __launch_bounds__(PYR_THREADS, 5) pyr_down_kernel(const PyrJob* __restrict__ jobs,
                                                                  const unsigned* __restrict__ tile_map,
                                                                  const uint8_t* const* frames,
                                                                  const uint8_t* src, int sp)
{
    // the next level's kernel (or the track kernel) may start its setup now;
    // the block's description (tables written before the chain started) is
    // read at once, this level's source only once the previous kernel is done
    griddep_launch_dependents();
    const Tile t = tile_at(jobs, tile_map, frames, src, sp, (int)blockIdx.x);
    const PyrJob& J = t.J;
    const int nx = (J.dW + PX - 1) / PX, ny = (J.dH + PY - 1) / PY;
    const int idx = t.local * PYR_THREADS + (int)threadIdx.x, lane = (int)threadIdx.x & 31;
    // (threads beyond the last repeat it without stores, for the shuffles)
    const bool active = idx < nx * ny;
    const int i = min(idx, nx * ny - 1), by = i / nx, bx = i - by * nx;
    const int ix = 2 * PX * bx, iy = 2 * PY * by - 2;
    const int nv = J.sW - ix;            // columns of the row from ix on
    const bool wide = ((reinterpret_cast<uintptr_t>(J.src) | (uintptr_t)J.sp) & 15u) == 0;
    griddep_wait();
    // rows iy .. iy + 10 (clamped), columns ix .. ix + 15; and, where no
    // neighbour in the warp has them, columns ix - 2, ix - 1 or ix + 16
    const bool left = lane == 0 && bx > 0, right = lane == 31 || bx == nx - 1;
    uint32_t m[PR][4], ed[PR];
    // Bytes beyond a row are any (replaced below) but never read from outside
    // the source: a level's rows have their pitch, a frame ends with its last row.
    auto row_at = [&](int r) { return J.src + (size_t)min(max(iy + r, 0), J.sH - 1) * J.sp; };
    const uint8_t* end = J.src + (t.copy0 ? (size_t)(J.sH - 1) * J.sp + J.sW : (size_t)J.sH * J.sp);
    if (wide && row_at(PR - 1) + ix + 16 <= end) {
#pragma unroll
        for (int r = 0; r < PR; ++r) {
            const uint4 v = src_load<uint4>(J, row_at(r) + ix);
            m[r][0] = v.x;
            m[r][1] = v.y;
            m[r][2] = v.z;
            m[r][3] = v.w;
        }
    } else {
        // rows of any alignment (a frame): the aligned words around the columns;
        // lo and hi are the first and the last word that lie in the frame, head and
        // tail its bytes before and after them
        const unsigned a0 = (unsigned)(reinterpret_cast<uintptr_t>(J.src) & 3u);
        const long long n = end - J.src, lo = -a0 & 3u, hi = n - (long long)((n + a0) & 3u) - 4;
        uint32_t head = 0, tail = 0;
#pragma unroll
        for (int b = 1; b < 4; ++b)
            if (lo - 4 + b >= 0) head |= (uint32_t)src_load<uint8_t>(J, J.src + lo - 4 + b) << (8 * b);
#pragma unroll
        for (int b = 0; b < 3; ++b)
            if (hi + 4 + b < n) tail |= (uint32_t)src_load<uint8_t>(J, J.src + hi + 4 + b) << (8 * b);
#pragma unroll
        for (int r = 0; r < PR; ++r) {
            const long long at = row_at(r) - J.src + ix;
            const unsigned a = (unsigned)(at + a0) & 3u;
            uint32_t w[5];
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                const long long o = at - a + 4 * q;
                w[q] = src_load<uint32_t>(J, J.src + min(max(o, lo), hi));
                w[q] = o < lo ? head : o > hi ? tail : w[q];     // (words beyond the tail hold no column of the row)
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) m[r][q] = __funnelshift_r(w[q], w[q + 1], 8 * a);
        }
    }
#pragma unroll
    for (int r = 0; r < PR; ++r) {
        const uint8_t* row = row_at(r);
        ed[r] = 0;
        if (left) ed[r] = src_byte(J, row, ix - 2) << 16 | src_byte(J, row, ix - 1) << 24;
        if (right) ed[r] |= src_byte(J, row, ix + 16);
    }
    if (nv < 16) {
        // the row ends within the 16 columns: its last byte beyond
        const int k = (nv - 1) & 3;
#pragma unroll
        for (int r = 0; r < PR; ++r) {
            const uint32_t lw = nv > 12 ? m[r][3] : nv > 8 ? m[r][2] : nv > 4 ? m[r][1] : m[r][0];
            const uint32_t rep = __byte_perm(lw, 0, 0x1111u * k);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int n = nv - 4 * q;
                if (n < 4) m[r][q] = __byte_perm(m[r][q], rep, n <= 0 ? 0x4444 : n == 1 ? 0x4440 : n == 2 ? 0x4410 : 0x4210);
            }
        }
    }
    if (t.copy0 && active) {
        // source rows 8 by .. 8 by + 7 and, of the last thread row, what is left
#pragma unroll
        for (int r = 2; r < PR; ++r) {
            const int y = iy + r;
            if (y < J.sH && (r < PR - 1 || by == ny - 1)) {
                uint8_t* d = checked(t.copy0 + (size_t)y * t.cp + ix, 16, t.copy0, (size_t)t.cp * J.sH, CK_PYR_DST);
                *reinterpret_cast<uint4*>(d) = make_uint4(m[r][0], m[r][1], m[r][2], m[r][3]);
                if (bx == nx - 1 && nv > 16) d[16] = (uint8_t)ed[r];
            }
        }
    }
    // horizontal sums of two outputs in the halves of a word (at most 16 * 255):
    // E = even columns, O = odd; output x of the pair is Ve[x-1] + 4 Vo[x-1] +
    // 6 Ve[x] + 4 Vo[x] + Ve[x+1]
    uint32_t h[5][4];
#pragma unroll
    for (int r = 0; r < PR; ++r) {
        uint32_t L = __shfl_up_sync(0xffffffffu, m[r][3], 1), R = __shfl_down_sync(0xffffffffu, m[r][0], 1);
        if (bx == 0)
            L = __byte_perm(m[r][0], 0, 0x0000);
        else if (lane == 0)
            L = ed[r];
        if (right) R = ed[r];
        uint32_t E[4], O[4], e[5], o[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            E[q] = m[r][q] & 0x00ff00ffu;
            O[q] = __byte_perm(m[r][q], 0, 0x4341);
        }
        e[0] = __byte_perm(L, E[0], 0x5452);
        o[0] = __byte_perm(L, O[0], 0x5453);
#pragma unroll
        for (int q = 1; q < 4; ++q) {
            e[q] = __byte_perm(E[q - 1], E[q], 0x5432);
            o[q] = __byte_perm(O[q - 1], O[q], 0x5432);
        }
        e[4] = __byte_perm(E[3], R & 0xffu, 0x5432);
#pragma unroll
        for (int q = 0; q < 4; ++q) h[r % 5][q] = e[q] + e[q + 1] + 6u * E[q] + 4u * (o[q] + O[q]);
        // rows r-4 .. r are output row (r - 4) / 2's (a sum is at most 16 * 16 * 255 + 128 < 2^16)
        if (r >= 4 && r % 2 == 0) {
            const int j = (r - 4) / 2, gy = PY * by + j;
            uint32_t v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[q] = h[(r + 1) % 5][q] + h[r % 5][q] + 0x00800080u + 6u * h[(r + 3) % 5][q] +
                       4u * (h[(r + 2) % 5][q] + h[(r + 4) % 5][q]);
            // (columns from dW on lie in the pitch's padding)
            if (active && gy < J.dH)
                *reinterpret_cast<uint2*>(checked(J.dst + (size_t)gy * J.dp + PX * bx, 8, J.dst, (size_t)J.dp * J.dH, CK_PYR_DST)) =
                    make_uint2(__byte_perm(v[0], v[1], 0x7531), __byte_perm(v[2], v[3], 0x7531));
        }
    }
}

namespace {
// ordinary or programmatic-dependent launch of a pyramid-family kernel
template <typename... KArgs, typename... Args>
cudaError_t launch_ex(void (*kern)(KArgs...), dim3 grid, int threads, cudaStream_t s, bool pdl,
                      Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}
}  // namespace

cudaError_t launch_pyr_down(const PyrJob* jobs_dev, const unsigned* tile_map_dev, int total, cudaStream_t s,
                            const uint8_t* const* frames, const uint8_t* src, int sp, bool pdl)
{
    if (total <= 0) return cudaSuccess;
    return launch_ex(pyr_down_kernel, dim3((unsigned)total), PYR_THREADS, s, pdl, jobs_dev, tile_map_dev,
                     frames, src, sp);
}

// Batched level-0 copy: frame s (contiguous, pitch W) -> pitched level 0.
__global__ void copy_frames_kernel(const uint8_t* const* __restrict__ frames,
                                   const CopyJob* __restrict__ jobs)
{
    griddep_launch_dependents();
    const CopyJob J = jobs[blockIdx.y];   // tables written before the chain started
    const uint8_t* src = frames[blockIdx.y];
    griddep_wait();
    const int n = J.W * J.H;
    const bool vec = ((J.W & 3) == 0) && ((reinterpret_cast<uintptr_t>(src) & 3) == 0);
    if (vec) {
        const int wpr = J.W / 4;
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < wpr * J.H; i += gridDim.x * blockDim.x) {
            const int y = i / wpr, c = i % wpr;
            const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(src + (size_t)y * J.W) + c);
            *reinterpret_cast<uint32_t*>(J.dst + (size_t)y * J.dp + 4 * c) = w;
        }
    } else {
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
            const int y = i / J.W, x = i % J.W;
            J.dst[(size_t)y * J.dp + x] = __ldg(src + i);
        }
    }
}

cudaError_t launch_copy_frames(const uint8_t* const* frames, const CopyJob* jobs, int njobs,
                               int max_bytes, cudaStream_t s, bool pdl)
{
    const int threads = 256;
    int bx = (max_bytes / 4 + threads - 1) / threads;
    if (bx > 256) bx = 256;
    if (bx < 1) bx = 1;
    return launch_ex(copy_frames_kernel, dim3((unsigned)bx, (unsigned)njobs), threads, s, pdl, frames, jobs);
}

// Mixed precision storage: FP16 (I, gx, gy, 0) per pixel, central differences
// halved (exact in FP16: multiples of 1/2 with |g| <= 127.5), 0 on the border.
__global__ void pack_kernel(const PackJob* __restrict__ jobs)
{
    griddep_launch_dependents();
    const PackJob J = jobs[blockIdx.y];   // written before the chain started
    griddep_wait();
    const int n = J.W * J.H;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int y = i / J.W, x = i % J.W;
        const uint8_t* row = J.src + (size_t)y * J.sp;
        const float I = row[x];
        float gx = 0.0f, gy = 0.0f;
        if (x > 0 && x < J.W - 1) gx = 0.5f * ((float)row[x + 1] - (float)row[x - 1]);
        if (y > 0 && y < J.H - 1) gy = 0.5f * ((float)row[x + J.sp] - (float)row[x - J.sp]);
        const __half2 ig = __floats2half2_rn(I, gx);
        const __half2 yz = __floats2half2_rn(gy, 0.0f);
        uint2 v;
        v.x = *reinterpret_cast<const uint32_t*>(&ig);
        v.y = *reinterpret_cast<const uint32_t*>(&yz);
        J.dst[i] = v;
    }
}

cudaError_t launch_pack(const PackJob* jobs, int njobs, int max_pixels, cudaStream_t s, bool pdl)
{
    const int threads = 256;
    int bx = (max_pixels + threads - 1) / threads;
    if (bx > 512) bx = 512;
    if (bx < 1) bx = 1;
    return launch_ex(pack_kernel, dim3((unsigned)bx, (unsigned)njobs), threads, s, pdl, jobs);
}

#ifdef GLT_CHECKED
unsigned check_flags_pyramid()
{
    unsigned v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_check_flags, sizeof(v));
    cudaMemcpyToSymbol(g_check_flags, &z, sizeof(z));
    return v;
}
#endif

}  // namespace glt

