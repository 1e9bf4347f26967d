// Phase table reweighted by hat-function weights, built on the device.
//
// The phase function with weights w is p_w = p h_w / Z(w): p the density of
// the unweighted table (constant (1/n) / (omu_j - omu_{j+1}) per unit cos
// theta on bin j, omu = 1 - cos theta at the levels j / n), h_w the linear
// interpolant of the weights w_k at the hat nodes mu_k = -1 + 2k/(n_w - 1)
// (h_w = sum_k w_k phi_k), Z(w) = int p h_w. One cluster of CTAs writes the
// packed blob of p_w's equal-probability table in the layout of
// table_format.h, so the walk, the camera density and the adjoint use it like
// any table:
//   1. each bin's mass p_j int h_w (h_w is linear between hat nodes, so
//      trapezoids piece by piece are exact), in double precision;
//   2. their running sum (a fixed-order block scan), Z(w) its total;
//   3. each level i: the bin whose running sum brackets i Z / n, and inside it
//      the root of the quadratic partial mass of the piece holding the level;
//   4. per-bin densities of the single-precision levels, the table mean and
//      the camera-density guide, computed with the same single-precision
//      operations as the host table builder's guide.
// Weights must be positive and finite; otherwise (or if single precision
// cannot hold the levels apart) the blob gets an invalid header, so a walk
// using it stops with MC_EFLAG_TABLE, and MC_EFLAG_NUMERIC is set.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "engine.h"
#include "table_format.h"

namespace mcx {
namespace {

namespace cg = cooperative_groups;

constexpr int WT_BLOCK = 1024;
constexpr int WT_CLUSTER = 8;   // CTAs of the one cluster (a portable cluster size)
constexpr unsigned FULL = 0xffffffffu;

// h_w at cos theta = mu: the two hats around mu
__device__ __forceinline__ double hw_at(const float *w, int n_w, double mu)
{
    const double t = (mu + 1.0) * (0.5 * (n_w - 1));
    int k = (int)floor(t);
    k = min(max(k, 0), n_w - 2);
    const double f = fmin(fmax(t - (double)k, 0.0), 1.0);
    return (double)w[k] * (1.0 - f) + (double)w[k + 1] * f;
}

// Pieces of bin [v_hi -> v_lo] in 1 - cos theta (v_hi > v_lo) between the
// hat nodes v_k = 2 - 2k/(n_w - 1) it contains, in order of decreasing v;
// fn(a, b, ha, hb) is called for each piece from a down to b.
template <class Fn>
__device__ __forceinline__ void for_pieces(const float *w, int n_w, double v_hi, double v_lo, Fn fn)
{
    const double step = 2.0 / (n_w - 1);
    // nodes strictly inside (v_lo, v_hi): k with 2 - k step in that range,
    // i.e. k in ((2 - v_hi) / step, (2 - v_lo) / step)
    int k0 = (int)floor((2.0 - v_hi) / step) + 1, k1 = (int)ceil((2.0 - v_lo) / step) - 1;
    k0 = max(k0, 0);
    k1 = min(k1, n_w - 1);
    double a = v_hi, ha = hw_at(w, n_w, 1.0 - v_hi);
    for (int k = k0; k <= k1; ++k) {
        const double vk = 2.0 - k * step;
        if (!(vk < a && vk > v_lo)) continue;
        const double hk = (double)w[k];
        if (!fn(a, vk, ha, hk)) return;
        a = vk;
        ha = hk;
    }
    fn(a, v_lo, ha, hw_at(w, n_w, 1.0 - v_lo));
}

// Inclusive scan in thread order of one double per thread over the first
// `warps` warps (warp scans, then the warps' totals); *total: their sum. Every
// thread of the CTA calls it. red: 32 doubles.
__device__ __forceinline__ double block_inclusive(double v, int warps, double *red, double *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < warps)
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(FULL, v, o);
            if (lane >= o) v += y;
        }
    __syncthreads();
    if (warp < warps && lane == 31) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double t = lane < warps ? red[lane] : 0.0;
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(FULL, t, o);
            if (lane >= o) t += y;
        }
        red[lane] = t;   // inclusive sums of the warps' totals
    }
    __syncthreads();
    *total = red[warps - 1];
    return warp > 0 && warp < warps ? v + red[warp - 1] : v;
}

// x of h(x) = ha + s x (x: distance below the piece's upper end a, length
// a - b) with integral ha x + s x^2 / 2 = rem, as 1 - cos theta.
__device__ __forceinline__ double piece_root(double a, double b, double ha, double hbv, double rem)
{
    const double s = (hbv - ha) / (a - b);
    const double x = 2.0 * rem / (ha + sqrt(fmax(ha * ha + 2.0 * s * rem, 0.0)));
    return fmin(fmax(a - x, b), a);
}

// Level i of p_w (in 1 - cos theta) inside bin j with remaining mass / p_j =
// rem, for a bin that hat nodes cut into pieces.
__device__ __noinline__ double level_pieces(double rem, double v_hi, double v_lo, const float *w, int n_w)
{
    double v = v_lo;
    for_pieces(w, n_w, v_hi, v_lo, [&](double a, double b, double ha, double hbv) {
        const double piece = 0.5 * (ha + hbv) * (a - b);
        if (rem <= piece) {
            v = piece_root(a, b, ha, hbv, rem);
            return false;
        }
        rem -= piece;
        return true;
    });
    return v;
}

__device__ __noinline__ double mass_pieces(double v_hi, double v_lo, const float *w, int n_w)
{
    double m = 0.0;
    for_pieces(w, n_w, v_hi, v_lo, [&](double a, double b, double ha, double hbv) {
        m += 0.5 * (ha + hbv) * (a - b);
        return true;
    });
    return m;
}

// X: the layout of an n-bin blob (the base blob's header must agree). One
// cluster of WT_CLUSTER CTAs: CTA r owns bins [r c, r c + c), c = n /
// WT_CLUSTER, and computes their widths, h_w at their edges, masses and levels;
// running sums are scanned per CTA and joined with the CTAs' totals, read
// through distributed shared memory, so all CTAs see identical edges and
// running masses. Dynamic shared memory: double ve[n + 1], cum[n + 1],
// mine[c + 1], hm[c + 1], red[32], part[4]; int kk[c + 1].
//
// Bound: the double-precision pipe (2 lanes per clock and SM; a warp's
// instruction holds it for 16 clocks) and the barriers. Bins that no hat node
// cuts, all but some n_w of them, take no division in their mass and three in
// their level; the searches compare integers. 4096 bins, 64 weights: 67 us (90
// us with every CTA scanning the whole table, h_w formed again at both edges of
// each use and divisions by the node spacing).
__global__ void __launch_bounds__(WT_BLOCK) weighted_table_kernel(const unsigned char *base, mc_table_header X,
                                                                  int n_w, const float *w, unsigned char *out,
                                                                  uint32_t *err)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), nr = (int)cluster.num_blocks();
    const int n = X.n_bins, c = n / nr;            // n_bins is a power of two, 64 at least
    const int r0 = rank * c, t = (int)threadIdx.x, warps = (c + 31) / 32;
    const int shift = 31 - __clz(c);
    extern __shared__ __align__(16) double sh[];
    const mc_table_header *hb = reinterpret_cast<const mc_table_header *>(base);
    mc_table_header *ho = reinterpret_cast<mc_table_header *>(out);
    double *ve = sh;
    double *cum = ve + n + 1;
    double *mine = cum + n + 1;
    double *hm = mine + c + 1;
    double *red = hm + c + 1;
    double *part = red + 32;   // [0], [1]: totals of the two scans, [2]: share of the mean, [3]: failure flag
    int *kk = reinterpret_cast<int *>(part + 4);
    bool bad = false;
    for (int k = t; k < n_w; k += blockDim.x) bad |= !(w[k] > 0.0f) || !isfinite(w[k]);
    if (hb->magic != MC_TABLE_MAGIC || hb->n_bins != n || hb->n_guide != X.n_guide || hb->off_omu != X.off_omu ||
        hb->off_pdf != X.off_pdf || hb->off_guide != X.off_guide || hb->total_bytes != X.total_bytes)
        bad = true;
    if (__syncthreads_or(bad)) {   // the same inputs in every CTA: all leave here together
        if (rank == 0 && t == 0) {
            atomicOr(err, MC_EFLAG_NUMERIC);
            ho->magic = 0u;    // walks using this blob stop with MC_EFLAG_TABLE
        }
        return;
    }
    const float *bpdf = reinterpret_cast<const float *>(base + hb->off_pdf);
    float *oo = reinterpret_cast<float *>(out + hb->off_omu);
    float *op = reinterpret_cast<float *>(out + hb->off_pdf);
    uint16_t *og = reinterpret_cast<uint16_t *>(out + hb->off_guide);
    const double inv_n = 1.0 / n;
    double total;

    // 0. the unweighted table's edges in double precision from its bin
    // densities (each bin holds 1/n): widths (1/n) / pdf_j summed from the
    // forward end, omu = 0, so every edge keeps the densities' relative
    // precision. Thread t scans the t-th bin from the CTA's forward end.
    double own = t < c ? inv_n / (double)bpdf[r0 + c - 1 - t] : 0.0;
    own = block_inclusive(own, warps, red, &total);
    if (t < c) mine[c - 1 - t] = own;
    if (t == 0) part[0] = total;
    cluster.sync();
    if (t < nr) {       // what lies forward of each CTA's bins
        double off = 0.0;
        for (int q = nr - 1; q > t; --q) off += *cluster.map_shared_rank(part, q);
        red[t] = off;
    }
    __syncthreads();
    for (int j = t; j < n; j += blockDim.x) {
        const int q = j >> shift;
        ve[j] = cluster.map_shared_rank(mine, q)[j - (q << shift)] + red[q];
    }
    if (t == 0) ve[n] = 0.0;
    cluster.sync();   // every CTA has read the sums: mine is free again

    // 1-2. h_w and the hat interval at this CTA's edges; bin masses p_j int h_w
    // and their running sum from mu = -1
    for (int j = t; j <= c; j += blockDim.x) {
        const double mu = 1.0 - ve[r0 + j];
        hm[j] = hw_at(w, n_w, mu);
        kk[j] = (int)floor((mu + 1.0) * (0.5 * (n_w - 1)));
    }
    __syncthreads();
    own = 0.0;
    if (t < c) {
        const double v_hi = ve[r0 + t], v_lo = ve[r0 + t + 1];
        const double m = kk[t] == kk[t + 1] ? 0.5 * (hm[t] + hm[t + 1]) * (v_hi - v_lo)
                                            : mass_pieces(v_hi, v_lo, w, n_w);
        own = (double)bpdf[r0 + t] * m;
    }
    own = block_inclusive(own, warps, red, &total);
    if (t < c) mine[t] = own;
    if (t == 0) part[1] = total;
    cluster.sync();
    if (t < nr) {
        double off = 0.0;
        for (int q = 0; q < t; ++q) off += cluster.map_shared_rank(part, q)[1];
        red[t] = off;
    }
    __syncthreads();
    for (int j = t; j < n; j += blockDim.x) {
        const int q = j >> shift;
        cum[j + 1] = cluster.map_shared_rank(mine, q)[j - (q << shift)] + red[q];
    }
    if (t == 0) cum[0] = 0.0;
    cluster.sync();   // every CTA has read the masses: mine is free again
    const double Z = cum[n];

    // 3-4. this CTA's levels r0 .. r0 + c (one solve each): the bin whose
    // running mass brackets i Z / n, then the root of the piece's quadratic
    // partial mass; the densities of its bins from the double levels (as the
    // host builder does), its share of the mean
    for (int i = t; i <= c; i += blockDim.x) {
        const int level = r0 + i;
        double v = level == 0 ? ve[0] : 0.0;
        if (level > 0 && level < n) {
            const double target = Z * ((double)level * inv_n);
            const long long key = __double_as_longlong(target);   // non-negative: ordered as integers
            int lo = 0, hi = n - 1;   // largest j with cum[j] <= target
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (__double_as_longlong(cum[mid]) <= key) lo = mid; else hi = mid - 1;
            }
            const int q = lo >> shift, jl = lo - (q << shift);
            const double *h = cluster.map_shared_rank(hm, q) + jl;
            const int *k = cluster.map_shared_rank(kk, q) + jl;
            const double ha = h[0], hbv = h[1], rem = (target - cum[lo]) / (double)bpdf[lo];
            if (k[0] == k[1])
                v = rem <= 0.5 * (ha + hbv) * (ve[lo] - ve[lo + 1]) ? piece_root(ve[lo], ve[lo + 1], ha, hbv, rem)
                                                                    : ve[lo + 1];
            else
                v = level_pieces(rem, ve[lo], ve[lo + 1], w, n_w);
        }
        mine[i] = v;
    }
    __syncthreads();
    double msum = 0.0;
    if (t < c) {
        const double vj = mine[t], vn = mine[t + 1], width = vj - vn;
        oo[r0 + t] = r0 + t == 0 ? 2.0f : (float)vj;
        if (!(width > 0.0)) bad = true;
        op[r0 + t] = (float)(inv_n / width);
        msum = 1.0 - 0.5 * (vj + vn);
    }
    if (rank == nr - 1 && t == 0) oo[n] = 0.0f;
    block_inclusive(msum, warps, red, &total);
    bad = __syncthreads_or(bad);
    if (t == 0) {
        part[2] = total;
        part[3] = bad ? 1.0 : 0.0;
    }
    __threadfence();   // the levels in global memory, before the guide reads them
    cluster.sync();
    bool any_bad = false;
    for (int q = 0; q < nr; ++q) any_bad |= __double_as_longlong(cluster.map_shared_rank(part, q)[3]) != 0;
    double mean = 0.0;
    if (rank == 0 && t == 0)
        for (int q = 0; q < nr; ++q) mean += cluster.map_shared_rank(part, q)[2];   // fixed order
    cluster.sync();   // no CTA leaves while others read its shares
    if (any_bad) {
        if (rank == 0 && t == 0) {
            atomicOr(err, MC_EFLAG_NUMERIC);
            ho->magic = 0u;
        }
        return;
    }

    // guide[c]: bin of the smallest float m with cell(m) >= c, where the
    // walk's lookup takes cell(m) = floor(fl(m + 1) (n_guide / 2)) and bin(m)
    // = the largest j with omu[j] >= fl(1 - m); this CTA's share of the cells
    float *levels = reinterpret_cast<float *>(cum);   // every CTA's, as stored
    for (int j = t; j <= n; j += blockDim.x) levels[j] = __ldcg(&oo[j]);
    __syncthreads();
    const int G = hb->n_guide;
    const int gc = (G + 1 + nr - 1) / nr, g0 = min(rank * gc, G + 1), g1 = min(g0 + gc, G + 1);
    const float half_g = 0.5f * (float)G;
    auto cell_of = [&](float m) { return (int)floorf((m + 1.0f) * half_g); };
    auto bin_of = [&](float m) {
        const float om = 1.0f - m;
        int lo = 0, hi = n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (levels[mid] >= om) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    auto key_of = [](float f) {
        const uint32_t b = __float_as_uint(f);
        return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
    };
    auto float_of = [](uint32_t k) {
        return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
    };
    for (int g = g0 + t; g < g1; g += blockDim.x) {
        float m;
        if (g == 0) {
            m = -1.0f;
        } else if (g == G) {
            m = 1.0f;
        } else {
            // fl(m + 1) is within 1.2e-7 of m + 1 and the product exact: the
            // answer lies within that of the cell's lower edge
            const float edge = (float)g / half_g - 1.0f;
            uint32_t lo = key_of(fmaxf(edge - 3e-7f, -1.0f)), hi = key_of(fminf(edge + 3e-7f, 1.0f));
            while (lo < hi) {
                const uint32_t mid = lo + (hi - lo) / 2;
                if (cell_of(float_of(mid)) >= g) hi = mid; else lo = mid + 1;
            }
            m = float_of(lo);
        }
        og[g] = (uint16_t)bin_of(m);
    }
    if (rank == 0 && t == 0) {
        mc_table_header h = *hb;
        h.g_table = (float)(mean * inv_n);
        *ho = h;
    }
}

}  // namespace

size_t weighted_table_smem(int n_bins)
{
    const size_t c = ((size_t)n_bins + WT_CLUSTER - 1) / WT_CLUSTER;
    return sizeof(double) * (2 * ((size_t)n_bins + 1) + 2 * (c + 1) + 32 + 4) + sizeof(int) * (c + 1);
}

cudaError_t launch_weighted_table(const unsigned char *base, int n_bins, int n_w, const float *w,
                                  unsigned char *out, uint32_t *err, cudaStream_t st)
{
    mc_table_header X;
    if (!mc_table_layout(n_bins, &X) || n_bins > kMaxWeightedBins) return cudaErrorInvalidValue;
    const size_t smem = weighted_table_smem(n_bins);
    cudaError_t e = cudaFuncSetAttribute(weighted_table_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(WT_CLUSTER);
    cfg.blockDim = dim3(WT_BLOCK);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = WT_CLUSTER;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, weighted_table_kernel, base, X, n_w, w, out, err);
}

}  // namespace mcx
