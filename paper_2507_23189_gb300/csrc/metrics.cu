// Image comparison metrics on the device (mc_image_metrics, include/mcmie.h):
// Sec. 3.1.4 normalises every image the same way (min-max to [0, 1] here),
// Table 3 compares images by RMSE and Pearson r, Table 4 compares radial
// profiles (means over rings about the image centre) zone by zone.
//
// Two launches over the pixels, spread over the whole chip:
//   scan_kernel   every pixel once: per image the extremes, the sum and the
//                 sum of each ring, all exact integers (a pixel's low and high
//                 32 bits summed apart), so their order does not matter
//   pair_kernel   every pixel once more, now that extremes and means are
//                 known: squared error and centred products of the normalised
//                 images in double precision, one row of partial sums per
//                 CTA; the last CTA to finish adds the rows in a fixed order
//                 and writes profiles, zone errors and correlations
// so the numbers do not depend on scheduling.
//
// What bounds them: GB300 issues 2 double-precision instructions per clock
// and SM, and one CTA per image or ring (the earlier layout: a division per
// pixel in each of n_r + 2 passes) left most SMs idle: a call on three
// 512 x 512 images with 32 rings took 4.87 ms, now 0.110 ms (the read-back
// of the numbers included). The scan uses no double-precision arithmetic but
// for pixels next to a ring's edge, the pair pass about 24 such instructions
// per pixel.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "../../include/mcmie.h"

namespace {

constexpr int MB = 256;        // threads per CTA, fixed: sums are ordered by it
constexpr int RUN = 8;         // consecutive pixels per scan thread: a ring is ~10 pixels wide at 512 x 512
                               // and 32 rings, so a run adds to one or two rings
constexpr int MAX_RINGS = 4096;
constexpr int SMEM_RINGS = 512;   // rings summed in shared memory first (26 KB); beyond, ring sums are spread
                                  // over so many addresses that L2 takes them directly
constexpr int MAX_PAIR_CTAS = 304;   // two per SM: a CTA's start and end cost about as much as 6 pixels a thread
constexpr unsigned FULL = 0xffffffffu;

struct Imgs {
    const long long *p[3];
};

typedef unsigned long long u64;

// The scan's results, zero before it runs. top: largest value and largest
// complement with the sign bit flipped (so that unsigned order is the order
// of the signed values and 0 is below all); sum of v = sum of its low words
// + 2^32 * sum of its (signed) high words.
struct Scan {
    u64 top_max[3], top_min[3];
    u64 tot_lo[3], tot_hi[3];
    unsigned int done;            // pair CTAs that have finished
    unsigned int pad;
};

struct Rings {
    u64 *lo, *hi;                 // [3][n_r]
    u64 *cnt;                     // [n_r]
};

// Ring of pixel (ix, iz): polar radius about the image centre in pixel units,
// n_r equal rings out to the half-diagonal (the radius itself goes last).
__device__ __forceinline__ int ring_of(int ix, int iz, int nx, int nz, double rho_max, int n_r)
{
    const double dx = ((double)ix + 0.5) - (double)nx / 2.0;
    const double dz = ((double)iz + 0.5) - (double)nz / 2.0;
    const double rho = sqrt(dx * dx + dz * dz);
    const double t = floor(rho / rho_max * (double)n_r);
    return t < (double)(n_r - 1) ? (int)t : n_r - 1;
}

// The same in single precision where that decides it: half-integer offsets
// below 2^23 are exact, the product is off by less than 4 2^-24 of itself
// (sum, square root, scale and product round once each), so at most 4096 x
// 2.4e-7 = 1e-3 of a ring; within that distance of an edge the
// double-precision form decides.
__device__ __forceinline__ int ring_fast(int ix, int iz, int nx, int nz, float scale, float margin, double rho_max,
                                         int n_r)
{
    const float dx = 0.5f * (float)(2 * ix + 1 - nx), dz = 0.5f * (float)(2 * iz + 1 - nz);
    const float t = sqrtf(dx * dx + dz * dz) * scale;
    const float f = floorf(t);
    if (t - f < margin || t - f > 1.0f - margin) return ring_of(ix, iz, nx, nz, rho_max, n_r);
    return min((int)f, n_r - 1);
}

__device__ __forceinline__ double half_diagonal(int nx, int nz)
{
    const double hx = (double)nx / 2.0, hz = (double)nz / 2.0;
    return sqrt(hx * hx + hz * hz);
}

__device__ __forceinline__ u64 flip(long long v) { return (u64)v ^ 0x8000000000000000ull; }

template <int NI>
__global__ void __launch_bounds__(MB) scan_kernel(Imgs im, int nx, int nz, int n_r, float scale, float margin,
                                                  Scan *sc, Rings R)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const bool local = n_r <= SMEM_RINGS;
    u64 *s_lo = reinterpret_cast<u64 *>(smem), *s_hi = s_lo + NI * n_r;
    unsigned int *s_cnt = reinterpret_cast<unsigned int *>(s_hi + NI * n_r);
    if (local) {
        for (int i = threadIdx.x; i < NI * n_r; i += MB) { s_lo[i] = 0ull; s_hi[i] = 0ull; }
        for (int i = threadIdx.x; i < n_r; i += MB) s_cnt[i] = 0u;
        __syncthreads();
    }
    const long long npix = (long long)nx * nz;
    const double rho_max = half_diagonal(nx, nz);
    u64 tmax[NI], tmin[NI], tlo[NI], thi[NI];
#pragma unroll
    for (int k = 0; k < NI; ++k) { tmax[k] = 0ull; tmin[k] = 0ull; tlo[k] = 0ull; thi[k] = 0ull; }
    for (long long r = blockIdx.x * (long long)MB + threadIdx.x; r * RUN < npix; r += (long long)gridDim.x * MB) {
        const long long i0 = r * RUN;
        const int len = (int)min((long long)RUN, npix - i0);
        int iz = (int)(i0 / nx), ix = (int)(i0 - (long long)iz * nx);
        int ring = -1;
        unsigned int c = 0;
        u64 lo[NI], hi[NI];
#pragma unroll
        for (int k = 0; k < NI; ++k) { lo[k] = 0ull; hi[k] = 0ull; }
        auto put = [&]() {      // the run's part in `ring`
#pragma unroll
            for (int k = 0; k < NI; ++k) {
                u64 *l = local ? s_lo + k * n_r + ring : R.lo + (size_t)k * n_r + ring;
                u64 *h = local ? s_hi + k * n_r + ring : R.hi + (size_t)k * n_r + ring;
                atomicAdd(l, lo[k]);
                atomicAdd(h, hi[k]);
                tlo[k] += lo[k];
                thi[k] += hi[k];
                lo[k] = 0ull;
                hi[k] = 0ull;
            }
            if (local) atomicAdd(&s_cnt[ring], c); else atomicAdd(&R.cnt[ring], (u64)c);
            c = 0;
        };
        for (int j = 0; j < len; ++j) {
            const int b = ring_fast(ix, iz, nx, nz, scale, margin, rho_max, n_r);
            if (b != ring) {
                if (c) put();
                ring = b;
            }
#pragma unroll
            for (int k = 0; k < NI; ++k) {
                const long long v = im.p[k][i0 + j];
                lo[k] += (u64)v & 0xffffffffull;
                hi[k] += (u64)(v >> 32);
                tmax[k] = max(tmax[k], flip(v));
                tmin[k] = max(tmin[k], ~flip(v));
            }
            ++c;
            if (++ix == nx) { ix = 0; ++iz; }
        }
        put();
    }
#pragma unroll
    for (int k = 0; k < NI; ++k) {
        for (int o = 16; o > 0; o >>= 1) {
            tmax[k] = max(tmax[k], __shfl_xor_sync(FULL, tmax[k], o));
            tmin[k] = max(tmin[k], __shfl_xor_sync(FULL, tmin[k], o));
            tlo[k] += __shfl_xor_sync(FULL, tlo[k], o);
            thi[k] += __shfl_xor_sync(FULL, thi[k], o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&sc->top_max[k], tmax[k]);
            atomicMax(&sc->top_min[k], tmin[k]);
            atomicAdd(&sc->tot_lo[k], tlo[k]);
            atomicAdd(&sc->tot_hi[k], thi[k]);
        }
    }
    if (local) {
        __syncthreads();
        for (int i = threadIdx.x; i < NI * n_r; i += MB) {
            if (s_lo[i]) atomicAdd(&R.lo[i], s_lo[i]);
            if (s_hi[i]) atomicAdd(&R.hi[i], s_hi[i]);
        }
        for (int i = threadIdx.x; i < n_r; i += MB)
            if (s_cnt[i]) atomicAdd(&R.cnt[i], (u64)s_cnt[i]);
    }
}

// An image's normalisation: v -> (v - mn) / (mx - mn) (0 for a constant image).
struct Norm {
    u64 mn;                       // smallest value
    double range, inv;            // largest - smallest and its reciprocal
};

__device__ __forceinline__ Norm norm_of(const Scan *sc, int k)
{
    Norm n;
    n.mn = ~sc->top_min[k];                          // still sign-flipped
    n.range = (double)(sc->top_max[k] - n.mn);
    n.inv = 1.0 / n.range;
    n.mn = n.mn ^ 0x8000000000000000ull;
    return n;
}

// d / range from the correctly rounded reciprocal and one residual step
// (Markstein, IBM J. Res. Dev. 34, 1990): within a last place of the quotient,
// and the rounded quotient itself in all of 4e8 random and near-midpoint pairs.
__device__ __forceinline__ double norm_px(long long v, const Norm &n)
{
    if (n.range == 0.0) return 0.0;
    const double d = (double)((u64)v - n.mn);
    const double q = d * n.inv;
    return fma(fma(-q, n.range, d), n.inv, q);
}

// (sum of v - cnt mn) / range: the sum of normalised values, from exact integers.
__device__ __forceinline__ double norm_sum(u64 lo, u64 hi, long long cnt, const Norm &n)
{
    if (n.range == 0.0) return 0.0;
    const __int128 s = (__int128)(long long)hi * ((__int128)1 << 32) + (__int128)lo - (__int128)cnt * (long long)n.mn;
    // non-negative, below 2^64 pixels x 2^26
    const u64 top = (u64)(s >> 32), low = (u64)s & 0xffffffffull;
    return fma((double)top, 4294967296.0, (double)low) / n.range;
}

// v[0..K) of the first `warps` warps summed in a fixed order (lanes, then
// warps); every thread gets the sums. One lane per value adds the warps' sums:
// each double-precision instruction holds an SM's pipe for 16 clocks a warp.
// red: (MB / 32 + 1) * K doubles.
template <int K>
__device__ __forceinline__ void block_sums(double (&v)[K], double *red, int warps = MB / 32)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (warp < warps) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(FULL, v[k], o);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < K; ++k) red[K + warp * K + k] = v[k];
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double t = 0.0;
        for (int q = 0; q < warps; ++q) t += red[K + q * K + threadIdx.x];
        red[threadIdx.x] = t;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = red[k];
}

// Images 1 .. NI-1 against image 0 (the reference); partials: [CTA][7] rows of
// squared error and reference product per pair, autos of pair 1, 2 and of the
// reference.
template <int NI>
__global__ void __launch_bounds__(MB) pair_kernel(Imgs im, long long npix, int n_r, Scan *sc, Rings R,
                                                  double *partials, double *out)
{
    __shared__ double red[(MB / 32 + 1) * 16];
    __shared__ bool last;
    __shared__ Norm s_nm[NI];
    __shared__ double s_mean[NI];
    if (threadIdx.x < NI) {     // one lane per image: three divisions each
        const int k = threadIdx.x;
        s_nm[k] = norm_of(sc, k);
        s_mean[k] = norm_sum(sc->tot_lo[k], sc->tot_hi[k], npix, s_nm[k]) / (double)npix;
    }
    __syncthreads();
    Norm nm[NI];
    double mean[NI];
#pragma unroll
    for (int k = 0; k < NI; ++k) {
        nm[k] = s_nm[k];
        mean[k] = s_mean[k];
    }
    double acc[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) acc[q] = 0.0;
    for (long long i = blockIdx.x * (long long)MB + threadIdx.x; i < npix; i += (long long)gridDim.x * MB) {
        const double vr = norm_px(im.p[0][i], nm[0]), dr = vr - mean[0];
        acc[6] = fma(dr, dr, acc[6]);
#pragma unroll
        for (int k = 1; k < NI; ++k) {
            const double va = norm_px(im.p[k][i], nm[k]), e = va - vr, da = va - mean[k];
            acc[3 * (k - 1)] = fma(e, e, acc[3 * (k - 1)]);
            acc[3 * (k - 1) + 1] = fma(da, dr, acc[3 * (k - 1) + 1]);
            acc[3 * (k - 1) + 2] = fma(da, da, acc[3 * (k - 1) + 2]);
        }
    }
    block_sums(acc, red);
    if (threadIdx.x == 0) {
        for (int q = 0; q < 7; ++q) partials[(size_t)blockIdx.x * 7 + q] = acc[q];
        __threadfence();
        last = atomicAdd(&sc->done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;

    // -------- the last CTA: totals of the rows, then everything of n_r size
    __threadfence();
#pragma unroll
    for (int q = 0; q < 7; ++q) acc[q] = 0.0;
    for (int r = threadIdx.x; r < (int)gridDim.x; r += MB)
        for (int q = 0; q < 7; ++q) acc[q] += __ldcg(&partials[(size_t)r * 7 + q]);
    const int row_warps = min((int)(gridDim.x + 31) / 32, MB / 32), ring_warps = min((n_r + 31) / 32, MB / 32);
    block_sums(acc, red, row_warps);
    double *prof = out + 13;   // [3][n_r]
    // sums over the rings that hold pixels: their number, profiles, the
    // profiles' squared differences and ring counts by zone, rings where
    // image 1 is closer than image 2
    double v[14];
#pragma unroll
    for (int q = 0; q < 14; ++q) v[q] = 0.0;
    for (int b = threadIdx.x; b < n_r; b += MB) {
        const long long cnt = (long long)R.cnt[b];
        double p[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int k = 0; k < NI; ++k)
            if (cnt) p[k] = norm_sum(R.lo[(size_t)k * n_r + b], R.hi[(size_t)k * n_r + b], cnt, nm[k]) / (double)cnt;
        for (int k = 0; k < 3; ++k) prof[(size_t)k * n_r + b] = p[k];
        if (!cnt) continue;
        const double ang = 180.0 * ((double)b + 0.5) / (double)n_r;
        v[0] += 1.0;
        v[1] += p[0];
#pragma unroll
        for (int k = 1; k < NI; ++k) {
            const double d = p[k] - p[0], d2 = d * d;
            v[1 + k] += p[k];
            if (ang < 30.0) v[4 + 3 * (k - 1)] += d2;
            else if (ang <= 120.0) v[5 + 3 * (k - 1)] += d2;
            else v[6 + 3 * (k - 1)] += d2;
        }
        if (ang < 30.0) v[10] += 1.0;
        else if (ang <= 120.0) v[11] += 1.0;
        else v[12] += 1.0;
        if (NI == 3 && fabs(p[1] - p[0]) < fabs(p[2] - p[0])) v[13] += 1.0;
    }
    block_sums(v, red, ring_warps);
    double c[5] = {0.0, 0.0, 0.0, 0.0, 0.0};   // centred profile products: reference, then cross and auto per pair
    for (int b = threadIdx.x; b < n_r; b += MB) {
        if (!R.cnt[b]) continue;
        const double dr = prof[b] - v[1] / v[0];
        c[0] += dr * dr;
#pragma unroll
        for (int k = 1; k < NI; ++k) {
            const double da = prof[(size_t)k * n_r + b] - v[1 + k] / v[0];
            c[2 * k - 1] += da * dr;
            c[2 * k] += da * da;
        }
    }
    block_sums(c, red, ring_warps);
    if (threadIdx.x < 2) {   // one thread per pair
        const int p = threadIdx.x;
        double *o = out + 6 * p;
        if (p + 1 < NI) {
            // p is a thread's own index: selects, not indexing, keep the sums in registers
            const double se = p ? acc[3] : acc[0], sar = p ? acc[4] : acc[1], saa = p ? acc[5] : acc[2];
            o[0] = sqrt(se / (double)npix);
            o[1] = (saa == 0.0 || acc[6] == 0.0) ? 0.0 : sar / sqrt(saa * acc[6]);
#pragma unroll
            for (int z = 0; z < 3; ++z) {
                const double s = p ? v[7 + z] : v[4 + z];
                o[2 + z] = v[10 + z] > 0.0 ? sqrt(s / v[10 + z]) : 0.0;
            }
            const double car = p ? c[3] : c[1], caa = p ? c[4] : c[2];
            o[5] = (v[0] == 0.0 || caa == 0.0 || c[0] == 0.0) ? 0.0 : car / sqrt(caa * c[0]);
        } else {
            for (int i = 0; i < 6; ++i) o[i] = 0.0;
        }
        if (p == 0) out[12] = (NI == 3 && v[0] > 0.0) ? v[13] / v[0] : 0.0;
    }
}

// Workspace: the scan's results, ring sums and counts (zeroed before the
// scan), then the pair pass's partial rows.
size_t up256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

extern "C" int mc_metrics_out_len(int n_r) { return (n_r < 1 || n_r > MAX_RINGS) ? 0 : 13 + 3 * n_r; }

extern "C" size_t mc_metrics_workspace_bytes(int n_r)
{
    if (n_r < 1 || n_r > MAX_RINGS) return 0;
    return up256(sizeof(Scan)) + up256(sizeof(u64) * 7 * (size_t)n_r) + up256(sizeof(double) * 7 * MAX_PAIR_CTAS);
}

namespace {

template <int NI>
cudaError_t launch_metrics(const Imgs &im, int nx, int nz, int n_r, Scan *sc, const Rings &R, double *partials,
                           double *out, cudaStream_t st)
{
    const long long npix = (long long)nx * nz;
    const double rho_max = sqrt(0.25 * nx * (double)nx + 0.25 * nz * (double)nz);
    const float scale = (float)(n_r / rho_max);
    const float margin = 1e-4f + 4e-7f * (float)n_r;   // the single-precision ring index's error, see ring_fast
    const long long runs = (npix + RUN - 1) / RUN;
    const unsigned scan_ctas = (unsigned)std::min<long long>((runs + MB - 1) / MB, 1216);
    const size_t smem = n_r <= SMEM_RINGS ? (sizeof(u64) * 2 * NI + sizeof(unsigned int)) * (size_t)n_r : 0;
    scan_kernel<NI><<<scan_ctas, MB, smem, st>>>(im, nx, nz, n_r, scale, margin, sc, R);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const unsigned pair_ctas = (unsigned)std::min<long long>((npix + MB - 1) / MB, MAX_PAIR_CTAS);
    pair_kernel<NI><<<pair_ctas, MB, 0, st>>>(im, npix, n_r, sc, R, partials, out);
    return cudaGetLastError();
}

}  // namespace

extern "C" mc_status mc_image_metrics(const int64_t *d_ref, const int64_t *d_a, const int64_t *d_b, int nx,
                                      int nz, int n_r, double *d_out, void *d_work, size_t work_bytes,
                                      void *stream)
{
    if (!d_ref || !d_a || !d_out || !d_work || nx < 1 || nz < 1 || (long long)nx * nz > (1ll << 26) ||
        n_r < 1 || n_r > MAX_RINGS || (reinterpret_cast<uintptr_t>(d_work) & 15) ||
        (reinterpret_cast<uintptr_t>(d_out) & 7) || (reinterpret_cast<uintptr_t>(d_ref) & 7) ||
        (reinterpret_cast<uintptr_t>(d_a) & 7) || (d_b && (reinterpret_cast<uintptr_t>(d_b) & 7)))
        return MC_ERR_ARG;
    if (work_bytes < mc_metrics_workspace_bytes(n_r)) return MC_ERR_NOMEM;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char *w = static_cast<unsigned char *>(d_work);
    Scan *sc = reinterpret_cast<Scan *>(w);
    w += up256(sizeof(Scan));
    Rings R;
    R.lo = reinterpret_cast<u64 *>(w);
    R.hi = R.lo + 3 * (size_t)n_r;
    R.cnt = R.hi + 3 * (size_t)n_r;
    w += up256(sizeof(u64) * 7 * (size_t)n_r);
    double *partials = reinterpret_cast<double *>(w);
    Imgs im;
    im.p[0] = reinterpret_cast<const long long *>(d_ref);
    im.p[1] = reinterpret_cast<const long long *>(d_a);
    im.p[2] = reinterpret_cast<const long long *>(d_b ? d_b : d_a);
    if (cudaMemsetAsync(d_work, 0, up256(sizeof(Scan)) + up256(sizeof(u64) * 7 * (size_t)n_r), st) != cudaSuccess)
        return MC_ERR_CUDA;
    const cudaError_t e = d_b ? launch_metrics<3>(im, nx, nz, n_r, sc, R, partials, d_out, st)
                              : launch_metrics<2>(im, nx, nz, n_r, sc, R, partials, d_out, st);
    return e == cudaSuccess ? MC_OK : MC_ERR_CUDA;
}
