// Preparation of a heterogeneous medium for the delta-tracking walk
// (mc_grid_prepare): per voxel mu_ext = k_ext n + mu_a (Eq. 17 per voxel)
// and the optical depth from the voxel's top face to the camera face
// y = +ly/2, which makes the camera transmittance of any collision exact
// with one gather; and the majorant of every cell of bx x by x bz voxels.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstring>

#include "engine.h"

namespace mcx {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// Double-precision conversions on the integer pipe: GB300's double-precision
// pipe takes 2 lanes per clock and SM, and with a conversion in, a product, a
// sum and a conversion out per voxel it set the time of the kernels below
// (84 % busy in column_kernel, 77 % in fold_kernel; 256^3 voxels: preparation
// 233 -> 61 us with the majorants in the same pass, fold 154 -> 120 us). Same
// results.
// (the rare cases are calls: a predicated conversion takes its turn in the
// pipe even where no lane needs it)
__device__ __noinline__ double to_double_any(float f) { return (double)f; }
__device__ __noinline__ float to_float_any(double d) { return (float)d; }

__device__ __forceinline__ double to_double(float f)
{
    const uint32_t u = __float_as_uint(f), m = u & 0x7FFFFFFFu;
    if (m - 0x00800000u >= 0x7F000000u) return to_double_any(f);   // zero, subnormal, infinity, NaN
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ float to_float(double d)   // round to nearest even
{
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t sign = hi & 0x80000000u, e = (hi >> 20) & 0x7FFu;
    if (((hi << 1) | lo) == 0u) return __uint_as_float(sign);
    // not a normal float with room for the rounding to carry into the exponent
    if (e - 897u >= 253u) return to_float_any(d);
    // hi:lo >> 29 without the sign, rebased, and the 29 bits below it
    const uint32_t top = (((hi & 0x7FFFFFFFu) << 3) | (lo >> 29)) - (896u << 23), rest = lo & 0x1FFFFFFFu;
    return __uint_as_float(sign | (top + ((rest > 0x10000000u || (rest == 0x10000000u && (top & 1u))) ? 1u : 0u)));
}

// One thread per (x, z) column, walking down from the camera face: writes
// (mu_ext, depth above) per voxel; consecutive threads touch consecutive x,
// so every row access is coalesced. The depth is summed in double: od + mu vy,
// product and sum rounded each. EXACT_VY: vy has at most 29 significant bits,
// so mu vy is exact and one FMA rounds the same once.
//
// On the way each thread keeps the largest mu_ext of the majorant cell it is
// in; where its column leaves the cell, the lanes in the same cell merge theirs
// and one of them merges with atomicMax on the float's bits, which order like
// the non-negative floats they are (maj starts at 0). The majorant takes the
// same single-precision fmaf as the voxels, so no voxel exceeds it.
//
// Bound: DRAM, 12 bytes a voxel (256^3: 29 us at the measured copy rate).
constexpr int COL_BLOCK = 64;    // small grids have few columns: more CTAs
constexpr int COL_AHEAD = 8;     // densities loaded ahead
template <bool EXACT_VY>
__global__ void __launch_bounds__(COL_BLOCK) column_kernel(const float *__restrict__ density, int gx, int gy, int gz,
                                                           int bx, int by, int bz, int mx, int my, float k_ext,
                                                           float mu_a, double vy, float2 *__restrict__ cells,
                                                           float *__restrict__ maj)
{
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x, cols = (long long)gx * gz;
    const bool in = t < cols;
    const long long tc = in ? t : cols - 1;     // a lane past the end reads the last column and writes nothing
    const int iz = (int)(tc / gx), ix = (int)(tc - (long long)iz * gx);
    const int cell = (iz / bz) * mx * my + ix / bx;             // of the column, without y
    const unsigned peers = __match_any_sync(FULL, cell);
    const bool leader = (threadIdx.x & 31) == __ffs((int)peers) - 1;
    const float *d = density + ((size_t)iz * gy) * gx + ix;
    float2 *o = cells + ((size_t)iz * gy) * gx + ix;
    double od = 0.0;
    float m = 0.f;
    int cy = (gy - 1) / by, cy0 = cy * by;      // current cell and its lowest voxel
    float now[COL_AHEAD], ahead[COL_AHEAD];
    auto load = [&](int top) {
#pragma unroll
        for (int k = 0; k < COL_AHEAD; ++k) ahead[k] = top >= k ? __ldcs(d + (size_t)(top - k) * gx) : 0.f;
    };
    load(gy - 1);
    for (int top = gy - 1; top >= 0; top -= COL_AHEAD) {
#pragma unroll
        for (int k = 0; k < COL_AHEAD; ++k) now[k] = ahead[k];
        load(top - COL_AHEAD);
#pragma unroll
        for (int k = 0; k < COL_AHEAD; ++k) {
            const int iy = top - k;
            if (iy < 0) break;
            const float mu = fmaf(k_ext, now[k], mu_a);
            if (in) o[(size_t)iy * gx] = make_float2(mu, to_float(od));
            od = EXACT_VY ? fma(to_double(mu), vy, od) : od + to_double(mu) * vy;
            m = fmaxf(m, mu);
            if (iy == cy0) {
                const unsigned top_bits = __reduce_max_sync(peers, __float_as_uint(m));
                if (leader) atomicMax(reinterpret_cast<int *>(&maj[cell + cy * mx]), (int)top_bits);
                m = 0.f;
                --cy;
                cy0 -= by;
            }
        }
    }
}

// One warp per voxel row along x, from its far end: every voxel before the
// one where a first flight ended takes the full voxel length vx of that
// flight's coefficient, gsum[ix] += vx * sum_{j > ix} ex[j]. Chunks of 32
// voxels with a warp suffix scan; rows with no entries cost their loads (their
// test is on the integer pipe).
__global__ void row_suffix_kernel(double *__restrict__ gsum, const double *__restrict__ ex, int gx, long long rows,
                                  double vx)
{
    const long long r = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    if (r >= rows) return;   // whole warps leave together
    const int lane = threadIdx.x & 31;
    const size_t base = (size_t)r * gx;
    double carry = 0.0;      // sum of ex beyond the current chunk
    for (int c = ((gx - 1) >> 5) << 5; c >= 0; c -= 32) {
        const int ix = c + lane;
        const double e = ix < gx ? ex[base + ix] : 0.0;
        const bool any = __any_sync(FULL, (__double_as_longlong(e) << 1) != 0);
        if (any) {
            double s = e;    // inclusive suffix within the chunk
            for (int o = 1; o < 32; o <<= 1) {
                const double t = __shfl_down_sync(FULL, s, o);
                if (lane + o < 32) s += t;
            }
            const double after = __shfl_down_sync(FULL, s, 1);
            const double total = __shfl_sync(FULL, s, 0);
            const double add = carry + (lane < 31 ? after : 0.0);
            if (ix < gx && add != 0.0) gsum[base + ix] += vx * add;
            carry += total;
        } else if (__double_as_longlong(carry) << 1 && ix < gx) {
            gsum[base + ix] += vx * carry;
        }
    }
}

// The same for the beam's own row, from its kRowCopies copies: one CTA, a
// voxel per thread, its copies loaded at once.
constexpr int BEAM_BLOCK = 256;
__global__ void __launch_bounds__(BEAM_BLOCK) beam_row_kernel(double *__restrict__ gsum, const double *__restrict__ exr,
                                                              int gx, double vx)
{
    __shared__ double part[BEAM_BLOCK / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double carry = 0.0;
    for (int c = (gx - 1) / BEAM_BLOCK * BEAM_BLOCK; c >= 0; c -= BEAM_BLOCK) {
        const int ix = c + threadIdx.x;
        double v[kRowCopies], s = 0.0;
#pragma unroll
        for (int k = 0; k < kRowCopies; ++k) v[k] = ix < gx ? exr[(size_t)k * gx + ix] : 0.0;
#pragma unroll
        for (int k = 0; k < kRowCopies; ++k) s += v[k];
        for (int o = 1; o < 32; o <<= 1) {   // inclusive suffix within the warp
            const double t = __shfl_down_sync(FULL, s, o);
            if (lane + o < 32) s += t;
        }
        __syncthreads();
        if (lane == 0) part[warp] = s;
        __syncthreads();
        double beyond = carry;
        for (int w = BEAM_BLOCK / 32 - 1; w > warp; --w) beyond += part[w];
        const double after = __shfl_down_sync(FULL, s, 1);
        if (ix < gx) gsum[ix] += vx * (beyond + (lane < 31 ? after : 0.0));
        for (int w = BEAM_BLOCK / 32 - 1; w >= 0; --w) carry += part[w];
    }
}

// One thread per (x, z) column, upward: a camera term A at a collision in
// voxel iy takes A times a full voxel height in every voxel above it (s1,
// summed below: run); its part in its own voxel is already in gsum. A warp
// whose columns have no source so far only rounds gsum (most columns lie off
// the beam), with no double-precision instruction; the rest is a call, which
// the compiler does not compute ahead for every voxel. Bound: DRAM, 20 bytes a
// voxel (256^3: 49 us at the measured copy rate).
__device__ __noinline__ double fold_voxel(double g, double a, double run, double k_vy, float *out)
{
    *out = to_float(g - k_vy * run);
    return run + a;
}

__global__ void __launch_bounds__(COL_BLOCK) fold_kernel(const double *__restrict__ gsum,
                                                         const double *__restrict__ s1, float *__restrict__ grad,
                                                         int gx, int gy, int gz, double k_vy)
{
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const unsigned lanes = __ballot_sync(FULL, t < (long long)gx * gz);   // those with a column
    if (t >= (long long)gx * gz) return;
    const int iz = (int)(t / gx), ix = (int)(t - (long long)iz * gx);
    const size_t base = (size_t)iz * gy * gx + ix;
    double run = 0.0;
    bool started = false;               // warp-uniform: some source at or below
    constexpr int AHEAD = 4;
    double g[AHEAD], a[AHEAD], ng[AHEAD], na[AHEAD];
    auto load = [&](int y0) {
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) {
            const bool ok = y0 + k < gy;
            ng[k] = ok ? __ldcs(gsum + base + (size_t)(y0 + k) * gx) : 0.0;
            na[k] = ok ? __ldcs(s1 + base + (size_t)(y0 + k) * gx) : 0.0;
        }
    };
    load(0);
    for (int y0 = 0; y0 < gy; y0 += AHEAD) {
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) { g[k] = ng[k]; a[k] = na[k]; }
        load(y0 + AHEAD);
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) {
            if (y0 + k >= gy) break;
            float *out = grad + base + (size_t)(y0 + k) * gx;
            started = started || __any_sync(lanes, (__double_as_longlong(a[k]) << 1) != 0);
            if (started) run = fold_voxel(g[k], a[k], run, k_vy, out);
            else *out = to_float(g[k]);
        }
    }
}

}  // namespace

namespace {
// One thread per box element (ix fastest): its copies summed in copy order
// into the voxel's own sums.
__global__ void box_merge_kernel(double *__restrict__ gsum, double *__restrict__ s1, const double *__restrict__ bgs,
                                 const double *__restrict__ bs1, int copies, size_t nbox, size_t bstride, int gx,
                                 int gy, int by0, int bz0, int bw)
{
    for (size_t b = blockIdx.x * (size_t)blockDim.x + threadIdx.x; b < nbox; b += (size_t)gridDim.x * blockDim.x) {
        double tg = 0.0, ts = 0.0;
        for (int c = 0; c < copies; ++c) {
            tg += bgs[(size_t)c * bstride + b];
            ts += bs1[(size_t)c * bstride + b];
        }
        const int ix = (int)(b % (size_t)gx);
        const size_t r = b / (size_t)gx;
        const int iy = by0 + (int)(r % (size_t)bw), iz = bz0 + (int)(r / (size_t)bw);
        const size_t v = ((size_t)iz * gy + iy) * gx + ix;
        gsum[v] += tg;
        s1[v] += ts;
    }
}
}  // namespace

cudaError_t launch_box_merge(double *gsum, double *s1, const double *bgs, const double *bs1, int copies,
                             size_t nbox, size_t bstride, int gx, int gy, int by0, int bz0, int bw, cudaStream_t st)
{
    box_merge_kernel<<<1024, 256, 0, st>>>(gsum, s1, bgs, bs1, copies, nbox, bstride, gx, gy, by0, bz0, bw);
    return cudaGetLastError();
}

cudaError_t launch_gradient_fold(double *gsum, const double *s1, const double *ex, const double *exr, float *grad,
                                 int gx, int gy, int gz, double k_ext, double vx, double vy, cudaStream_t st)
{
    cudaError_t e;
    if (ex) {
        const long long rows = (long long)gy * gz;
        row_suffix_kernel<<<(unsigned)((rows * 32 + 255) / 256), 256, 0, st>>>(gsum, ex, gx, rows, vx);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (exr) {
        beam_row_kernel<<<1, BEAM_BLOCK, 0, st>>>(gsum + ((size_t)(gz / 2) * gy + gy / 2) * gx, exr, gx, vx);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const long long cols = (long long)gx * gz;
    fold_kernel<<<(unsigned)((cols + COL_BLOCK - 1) / COL_BLOCK), COL_BLOCK, 0, st>>>(gsum, s1, grad, gx, gy, gz,
                                                                                    k_ext * vy);
    return cudaGetLastError();
}

cudaError_t launch_grid_prepare(const float *density, int gx, int gy, int gz, int bx, int by, int bz,
                                float k_ext, float mu_a, double vy, float2 *cells, float *maj,
                                cudaStream_t st)
{
    const int mx = (gx + bx - 1) / bx, my = (gy + by - 1) / by, mz = (gz + bz - 1) / bz;
    cudaError_t e = cudaMemsetAsync(maj, 0, sizeof(float) * (size_t)mx * my * mz, st);
    if (e != cudaSuccess) return e;
    const long long cols = (long long)gx * gz;
    const unsigned ctas = (unsigned)((cols + COL_BLOCK - 1) / COL_BLOCK);
    // a product of 24 and 29 significant bits fits a double's 53
    unsigned long long bits;
    static_assert(sizeof bits == sizeof vy, "");
    std::memcpy(&bits, &vy, sizeof bits);
    auto kern = (bits & 0xFFFFFFull) == 0 ? column_kernel<true> : column_kernel<false>;
    kern<<<ctas, COL_BLOCK, 0, st>>>(density, gx, gy, gz, bx, by, bz, mx, my, k_ext, mu_a, vy, cells, maj);
    return cudaGetLastError();
}

}  // namespace mcx
