// kernels.cu -- the row-pointer scan, the region vectors, the sampled-noise
// kernels and the per-pair FP64 kernel.
//
// FP64 builds are made by walk_fp64.cu; rows_fp64 here builds those whose
// tables do not fit it (a window box of more than 2048 targets): one warp per
// row evaluates every factor of every candidate pair.
// Per row:
//   1. interval image [m_lo, m_hi] of f over the cell (table lookups + sums)
//   2. per dimension, a window of target cells outside of which every upper
//      factor is below cutoff/2 (Sec. 4.4: entries whose upper bound is
//      negligible are not stored), trimmed to the targets that pass alone
//   3. the window box is enumerated in C order, lanes test up >= cutoff and
//      the warp compacts the kept targets with ballot/popc
//   4. per-row terms: the out-of-domain sink bounds (Remark 4.1), the
//      truncated mass and the row-sum checks of Def. 3.1, combined in FP64.
// The count pass runs 1-4 without storing pairs; a scan turns the counts into
// row pointers; the emit pass repeats 1-3 and writes the CSR pairs.
#include <cuda_runtime.h>

#include <algorithm>
#include <math.h>
#include <stdint.h>

#include "impact_desc.h"
#include "kernels.h"
#include "mc_keys.cuh"
#include "rowmath.cuh"
#include "scan.cuh"
#include "sound_fp32.cuh"

namespace {

using namespace mckeys;
using namespace rowmath;
using namespace rowscan;

constexpr int kWarpsPerBlock = 8;
constexpr int kThreads = kWarpsPerBlock * 32;
constexpr int kTab = IMPACT_TABLE_MAX;   // staged factor entries per row (all dims)

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---------------------------------------------------------------------------
// FP64 plain row kernel: every factor of every candidate pair in FP64
// ---------------------------------------------------------------------------

// Upper factor of target cell t of dimension d.
__device__ __forceinline__ double up64(const ImpactDim &g, const double *E, int t, double mlo,
                                       double mhi)
{
    double c = E[t], e = E[t + 1];
    return g64(c, e, clampd(0.5 * (c + e), mlo, mhi), g.inv_s);
}

__device__ __forceinline__ double lo64(const ImpactDim &g, const double *E, int t, double mlo,
                                       double mhi)
{
    double c = E[t], e = E[t + 1];
    return fmin(g64(c, e, mlo, g.inv_s), g64(c, e, mhi, g.inv_s));
}

struct WarpSm64 {
    double U[kTab];
    double mlo[IMPACT_MAX_DIM], mhi[IMPACT_MAX_DIM];
    double SW[IMPACT_MAX_DIM], O[IMPACT_MAX_DIM];
    double gin_max[IMPACT_MAX_DIM], gin_min[IMPACT_MAX_DIM];
    int a[IMPACT_MAX_DIM], w[IMPACT_MAX_DIM], cum[IMPACT_MAX_DIM];
    int ta[IMPACT_MAX_DIM], tw[IMPACT_MAX_DIM];
};

template <bool EMIT>
__global__ void __launch_bounds__(kThreads)
rows_fp64(const ImpactDesc *__restrict__ Dp, int64_t row_begin, int64_t row_end,
          int64_t *__restrict__ row_ptr, int32_t *__restrict__ out_col,
          double *__restrict__ out_lo, double *__restrict__ out_up,
          double *__restrict__ sink_lo, double *__restrict__ sink_up,
          double *__restrict__ trunc, uint32_t *__restrict__ flags,
          uint32_t *__restrict__ status, int64_t capacity, int64_t total_at)
{
    __shared__ WarpSm64 sm_all[kWarpsPerBlock];
    const ImpactDesc &D = *Dp;
    const int lane = threadIdx.x & 31;
    WarpSm64 &S = sm_all[threadIdx.x >> 5];
    const int n = D.n;
    const double cut = D.cutoff;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const unsigned lt = lanemask_lt();
    if (EMIT && capacity >= 0 && row_ptr[total_at] > capacity) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(status, IMPACT_STATUS_CAPACITY);
        return;
    }

    for (int64_t row = row_begin + warp0; row < row_end; row += nwarps) {
        int idx[IMPACT_MAX_DIM];
        int j;
        decode_row(D, row, idx, j);
        if (lane < n) {
            const ImpactDim &g = D.dim[lane];
            double mlo, mhi;
            image_dim<false>(D, row, idx, j, lane, mlo, mhi);
            int a, b;
            window_dim(g, mlo, mhi, a, b);
            S.mlo[lane] = mlo;
            S.mhi[lane] = mhi;
            S.a[lane] = a;
            S.w[lane] = b - a + 1;
            if (!EMIT) {   // in-domain mass at the three points (sink)
                double mid = 0.5 * (g.lo + g.hi);
                S.gin_max[lane] = g64(g.lo, g.hi, clampd(mid, mlo, mhi), g.inv_s);
                S.gin_min[lane] = fmin(g64(g.lo, g.hi, mlo, g.inv_s), g64(g.lo, g.hi, mhi, g.inv_s));
            }
        }
        __syncwarp();
        int total = 0;
        for (int d = 0; d < n; ++d) {
            if (lane == 0) S.cum[d] = total;
            total += S.w[d];
        }
        __syncwarp();
        // upper factors of the window (used only to trim the windows and for
        // the truncated-mass sums; the pairs below recompute every factor),
        // staged when they fit, else evaluated again where they are read
        const bool staged = total <= kTab;
        if (staged) {
            for (int e = lane; e < total; e += 32) {
                int d = 0;
                while (d + 1 < n && e >= S.cum[d + 1]) ++d;
                const ImpactDim &g = D.dim[d];
                S.U[e] = up64(g, D.edges + g.edge_off, S.a[d] + e - S.cum[d], S.mlo[d], S.mhi[d]);
            }
        }
        __syncwarp();
        bool empty = false;
        for (int d = 0; d < n; ++d) {
            const int base = S.cum[d], W = S.w[d];
            const ImpactDim &gd = D.dim[d];
            auto Uw = [&](int t) {
                return staged ? S.U[base + t]
                              : up64(gd, D.edges + gd.edge_off, S.a[d] + t, S.mlo[d], S.mhi[d]);
            };
            int first = -1, last = -1;
            for (int c0 = 0; c0 < W; c0 += 32) {
                int t = c0 + lane;
                bool pass = t < W && Uw(t) >= cut;
                unsigned bal = __ballot_sync(0xffffffffu, pass);
                if (bal) {
                    if (first < 0) first = c0 + __ffs(bal) - 1;
                    last = c0 + 31 - __clz(bal);
                }
            }
            double sw = 0.0, ow = 0.0;
            for (int c0 = 0; c0 < W; c0 += 32) {
                int t = c0 + lane;
                if (t < W) {
                    double v = Uw(t);
                    if (first >= 0 && t >= first && t <= last) sw += v;
                    else ow += v;
                }
            }
            sw = warp_sum_d(sw);
            ow = warp_sum_d(ow);
            if (lane == 0) {
                const ImpactDim &g = D.dim[d];
                const double *E = D.edges + g.edge_off;
                const int a = S.a[d], b = a + W - 1;
                double O = ow;
                if (a > 0) O += g64(E[0], E[a], S.mlo[d], g.inv_s);
                if (b < g.N - 1) O += g64(E[b + 1], E[g.N], S.mhi[d], g.inv_s);
                S.O[d] = O;
                S.SW[d] = sw;
                S.ta[d] = first < 0 ? a : a + first;
                S.tw[d] = first < 0 ? 0 : last - first + 1;
            }
            empty |= (first < 0);
        }
        __syncwarp();

        double drop = 0.0, slo = 0.0, sup = 0.0;
        int64_t cnt = 0, out_base = 0, out_end = 0, written = 0;
        if (EMIT) {
            out_base = row_ptr[row];
            out_end = row_ptr[row + 1];
        }
        if (!empty) {
            int64_t K = 1;
            for (int d = 0; d < n; ++d) K *= S.tw[d];
            int tt[IMPACT_MAX_DIM], sd[IMPACT_MAX_DIM];
            uint32_t q = (uint32_t)lane, qs = 32u;
            for (int d = n - 1; d >= 0; --d) {
                uint32_t W = (uint32_t)S.tw[d];
                tt[d] = (int)(q % W);
                q /= W;
                sd[d] = (int)(qs % W);
                qs /= W;
            }
            for (int64_t kb = 0; kb < K; kb += 32) {
                bool valid = (kb + lane < K);
                bool keep = false;
                double uv = 1.0, lv = 1.0;
                int cv = 0;
                if (valid) {
                    for (int d = 0; d < n; ++d) {
                        const ImpactDim &g = D.dim[d];
                        int t = S.ta[d] + tt[d];
                        uv *= up64(g, D.edges + g.edge_off, t, S.mlo[d], S.mhi[d]);
                        cv += t * g.stride;
                    }
                    keep = uv >= cut;
                    if (keep) {
                        for (int d = 0; d < n; ++d) {
                            const ImpactDim &g = D.dim[d];
                            lv *= lo64(g, D.edges + g.edge_off, S.ta[d] + tt[d], S.mlo[d], S.mhi[d]);
                        }
                    }
                }
                unsigned bal = __ballot_sync(0xffffffffu, keep);
                if (EMIT) {
                    if (keep) {
                        int64_t p = out_base + written + __popc(bal & lt);
                        if (p < out_end) {
                            out_col[p] = cv;
                            out_lo[p] = lv;
                            out_up[p] = uv;
                        }
                    }
                    written += __popc(bal);
                } else {
                    cnt += __popc(bal);
                    if (keep) {
                        slo += lv;
                        sup += uv;
                    } else if (valid) {
                        drop += uv;
                    }
                }
                int carry = 0;
                for (int d = n - 1; d >= 0; --d) {
                    int t = tt[d] + sd[d] + carry;
                    carry = t >= S.tw[d];
                    tt[d] = carry ? t - S.tw[d] : t;
                }
            }
        }
        if (EMIT && lane == 0 && out_base + written != out_end)
            atomicOr(status, IMPACT_STATUS_EMIT_MISMATCH);
        if (!EMIT) {
            double dsum = warp_sum_d(drop);
            double lsum = warp_sum_d(slo);
            double usum = warp_sum_d(sup);
            if (lane == 0) {
                double outside = 0.0;
                for (int d = 0; d < n; ++d) {
                    double t = S.O[d];
                    for (int k = 0; k < d; ++k) t *= S.SW[k];
                    for (int k = d + 1; k < n; ++k) t *= S.SW[k] + S.O[k];
                    outside += t;
                }
                double pmax = 1.0, pmin = 1.0;
                for (int d = 0; d < n; ++d) {
                    pmax *= S.gin_max[d];
                    pmin *= S.gin_min[d];
                }
                double sl = 1.0 - pmax, su = 1.0 - pmin;
                double tr = outside + dsum;
                row_ptr[row] = cnt;
                sink_lo[row] = sl;
                sink_up[row] = su;
                trunc[row] = tr;
                if (flags) {
                    uint32_t f = 0;
                    if (lsum + sl > 1.0 + 1e-12) f |= 0x1u;
                    if (usum + su + tr < 1.0 - 1e-12) f |= 0x2u;
                    flags[row] = f;
                    if (f) atomicOr(status, IMPACT_STATUS_UNSOUND);
                }
            }
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// Exclusive scan of the per-row counts (in place in row_ptr): tile sums, then
// every tile adds up the sums before it and applies its own scan. One tile
// needs no sums; beyond kScanSelf tiles a pass over the sums comes between. The
// builds' row-terms kernels do the first pass of few tiles in blocks of their own:
// one launch less, builds of 4092 rows 93 -> 83 us (with the status block's
// memset). With several tiles per SM they hold the terms up instead (24 random
// systems, 0.9M rows: 5.152 -> 5.159 ms).
// ---------------------------------------------------------------------------

constexpr int kScanThreads = 1024;
constexpr int64_t kScanSelf = 4 * kScanThreads;   // tile sums a block adds up itself
constexpr int64_t kScanHead = 152;                // tiles of another kernel's blocks: one per SM

__global__ void __launch_bounds__(kScanThreads) scan_tiles(const int64_t *__restrict__ v,
                                                           int64_t n, int64_t *__restrict__ tsum)
{
    tile_sum<kScanThreads>(v, n, blockIdx.x, tsum);
}

__global__ void __launch_bounds__(kScanThreads) scan_sums(int64_t *__restrict__ tsum, int64_t nt)
{
    __shared__ int64_t sh[32];
    int64_t carry = 0;
    for (int64_t b = 0; b < nt; b += kScanThreads) {
        int64_t i = b + threadIdx.x;
        int64_t v = i < nt ? tsum[i] : 0;
        int64_t total;
        int64_t ex = block_excl_scan<kScanThreads>(v, sh, total);
        if (i < nt) tsum[i] = carry + ex;
        carry += total;
    }
}

// SELF: toff holds the tiles' sums (unused by the first tile), else their
// offsets.
template <bool SELF>
__global__ void __launch_bounds__(kScanThreads) scan_apply(int64_t *__restrict__ v, int64_t n,
                                                           const int64_t *__restrict__ toff,
                                                           int64_t *__restrict__ also)
{
    __shared__ int64_t sh[32];
    int64_t before = 0;
    if (SELF) {
        int64_t s = 0;
        for (int i = threadIdx.x; i < blockIdx.x; i += kScanThreads) s += toff[i];
        if (blockIdx.x > 0) block_excl_scan<kScanThreads>(s, sh, before);
    } else {
        before = toff[blockIdx.x];
    }
    tile_apply<kScanThreads>(v, n, blockIdx.x, before, blockIdx.x == gridDim.x - 1, also);
}

// ---------------------------------------------------------------------------
// target / avoid regions (Sec. 3.1, Alg. 1, Remark 4.1)
// ---------------------------------------------------------------------------

using impact::RegionBoxes;
using impact::RowOutputs;

__global__ void __launch_bounds__(256)
label_cells(RegionBoxes B, int64_t total, uint8_t *__restrict__ labels)
{
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < total;
         c += (int64_t)gridDim.x * blockDim.x) {
        int idx[IMPACT_MAX_DIM];
        int64_t rest = c;
        for (int d = B.n - 1; d >= 0; --d) {
            idx[d] = (int)(rest % B.cells[d]);
            rest /= B.cells[d];
        }
        uint8_t lab = 0;
        for (int b = 0; b < B.count; ++b) {
            bool in = true;
            for (int d = 0; d < B.n; ++d)
                in = in && idx[d] >= B.first[b][d] && idx[d] <= B.last[b][d];
            if (in) lab = b >= B.n_target ? 2 : (lab == 0 ? 1 : lab);
        }
        labels[c] = lab;
    }
}

// FP32 interval of (p - m') / (sigma sqrt2) for every m' within dm of m: the
// FP64 evaluation (relative error below 2^-49 with the rounded 1/(sigma
// sqrt2)) widened by that error and by dm, then rounded outward to FP32.
__device__ __forceinline__ void arg_iv(double p, double m, double dm, double inv_s, float &lo,
                                       float &hi)
{
    const double x = (p - m) * inv_s;
    const double w = dm * inv_s;
    const double e = (fabs(x) + w) * 0x1p-49 + w;
    lo = __double2float_rd(x - e);
    hi = __double2float_ru(x + e);
}

// Bounds of one factor g(c, e; m), the mass of [c, e] around a mean m known
// to within dm: FP64 round-to-nearest (plain), or the FP32 outward bounds of
// sound_fp32.cuh (sound).
template <bool SOUND>
__device__ __forceinline__ double g_up(double c, double e, double m, double dm, double inv_s)
{
    if (!SOUND) return g64(c, e, m, inv_s);
    float acl, ach, ael, aeh;
    arg_iv(c, m, dm, inv_s, acl, ach);
    arg_iv(e, m, dm, inv_s, ael, aeh);
    return (double)sound::mass_hi(acl, ach, ael, aeh);
}
template <bool SOUND>
__device__ __forceinline__ double g_dn(double c, double e, double m, double inv_s)
{
    if (!SOUND) return g64(c, e, m, inv_s);
    float acl, ach, ael, aeh;
    arg_iv(c, m, 0.0, inv_s, acl, ach);
    arg_iv(e, m, 0.0, inv_s, ael, aeh);
    return (double)sound::mass_lo(acl, ach, ael, aeh);
}

// Largest factor over m in [mlo, mhi] (at the clamped midpoint of [c, e],
// whose rounding dm the sound bound covers) and the smallest (at an end).
template <bool SOUND>
__device__ __forceinline__ double f_max(double c, double e, double mlo, double mhi, double inv_s)
{
    const double mid = 0.5 * (c + e);
    const double m = clampd(mid, mlo, mhi);
    const double dm = (m == mid) ? fabs(mid) * 0x1p-52 : 0.0;
    return g_up<SOUND>(c, e, m, dm, inv_s);
}
template <bool SOUND>
__device__ __forceinline__ double f_min(double c, double e, double mlo, double mhi, double inv_s)
{
    return fmin(g_dn<SOUND>(c, e, mlo, inv_s), g_dn<SOUND>(c, e, mhi, inv_s));
}

template <bool SOUND>
__device__ __forceinline__ double mul_up(double a, double b) { return SOUND ? __dmul_ru(a, b) : a * b; }
template <bool SOUND>
__device__ __forceinline__ double mul_dn(double a, double b) { return SOUND ? __dmul_rd(a, b) : a * b; }
template <bool SOUND>
__device__ __forceinline__ double add_up(double a, double b) { return SOUND ? __dadd_ru(a, b) : a + b; }
template <bool SOUND>
__device__ __forceinline__ double add_dn(double a, double b) { return SOUND ? __dadd_rd(a, b) : a + b; }

// Largest and smallest factor of a block of cells [first, last] of dimension d
// over the image: the block's own (one relaxation), or the sums of its cells'
// (the paper's sums: the sum over a box's cells of a product of per-dimension
// factors equals the product of the per-dimension sums). first < 0: the whole
// domain as one block.
template <bool SOUND>
__device__ __forceinline__ double2 block_factor(const ImpactDim &g, const double *E, int first,
                                                int last, bool cell_sum, double mlo, double mhi)
{
    if (first < 0 || !cell_sum) {
        const double c = first < 0 ? g.lo : E[first], e = first < 0 ? g.hi : E[last + 1];
        return make_double2(f_max<SOUND>(c, e, mlo, mhi, g.inv_s),
                            f_min<SOUND>(c, e, mlo, mhi, g.inv_s));
    }
    double fu = 0.0, fl = 0.0;
    if (SOUND) {
        for (int i = first; i <= last; ++i) {
            fu = add_up<SOUND>(fu, f_max<SOUND>(E[i], E[i + 1], mlo, mhi, g.inv_s));
            fl = add_dn<SOUND>(fl, f_min<SOUND>(E[i], E[i + 1], mlo, mhi, g.inv_s));
        }
        return make_double2(fu, fl);
    }
    // plain: erfc once per edge and image end, shared by the cells beside it
    double c = E[first], x0 = (c - mlo) * g.inv_s, x1 = (c - mhi) * g.inv_s;
    double f0 = erfc(fabs(x0)), f1 = erfc(fabs(x1));
    for (int i = first; i <= last; ++i) {
        const double e = E[i + 1], y0 = (e - mlo) * g.inv_s, y1 = (e - mhi) * g.inv_s;
        const double h0 = erfc(fabs(y0)), h1 = erfc(fabs(y1));
        const double lo = mass64(x0, f0, y0, h0), hi = mass64(x1, f1, y1, h1);
        const double mid = 0.5 * (c + e);
        fu += mid < mlo ? lo : mid > mhi ? hi : g64(c, e, mid, g.inv_s);
        fl += fmin(lo, hi);
        c = e;
        x0 = y0;
        x1 = y1;
        f0 = h0;
        f1 = h1;
    }
    return make_double2(fu, fl);
}

// The row's four vectors from its blocks' factors, f(b, d) for b = -1 (the
// domain) and the boxes: the sink (Remark 4.1), then the products over the
// dimensions summed over the boxes.
template <bool SOUND, typename F>
__device__ __forceinline__ void region_vectors(const RegionBoxes &B, int n, F f, int64_t row,
                                               double *r_lo, double *r_up, double *a_lo,
                                               double *a_up)
{
    double rl = 0.0, ru = 0.0, xl = 0.0, xu = 0.0;
    for (int b = -1; b < B.count; ++b) {
        double pu = 1.0, pl = 1.0;
        for (int d = 0; d < n; ++d) {
            const double2 v = f(b, d);
            pu = mul_up<SOUND>(pu, v.x);
            pl = mul_dn<SOUND>(pl, v.y);
        }
        if (b < 0) {
            xl = SOUND ? fmax(__dsub_rd(1.0, pu), 0.0) : 1.0 - pu;
            xu = SOUND ? fmin(__dsub_ru(1.0, pl), 1.0) : 1.0 - pl;
        } else if (b < B.n_target) {
            rl = add_dn<SOUND>(rl, pl);
            ru = add_up<SOUND>(ru, pu);
        } else {
            xl = add_dn<SOUND>(xl, pl);
            xu = add_up<SOUND>(xu, pu);
        }
    }
    r_lo[row] = rl;
    r_up[row] = ru;
    a_lo[row] = xl;
    a_up[row] = xu;
}

// Rows whose images are (nearly) all distinct: one thread per row evaluates
// its blocks' factors.
template <bool SOUND>
__global__ void __launch_bounds__(128)
region_rows(const ImpactDesc *__restrict__ Dp, int64_t rows, RegionBoxes B, bool cell_sum,
            double *__restrict__ r_lo, double *__restrict__ r_up, double *__restrict__ a_lo,
            double *__restrict__ a_up)
{
    const ImpactDesc &D = *Dp;
    const int n = D.n;
    for (int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; row < rows;
         row += (int64_t)gridDim.x * blockDim.x) {
        int idx[IMPACT_MAX_DIM];
        int j;
        decode_row(D, row, idx, j);
        double mlo[IMPACT_MAX_DIM], mhi[IMPACT_MAX_DIM];
        for (int d = 0; d < n; ++d) image_dim<SOUND>(D, row, idx, j, d, mlo[d], mhi[d]);
        auto f = [&](int b, int d) {
            const ImpactDim &g = D.dim[d];
            return block_factor<SOUND>(g, D.edges + g.edge_off, b < 0 ? -1 : B.first[b][d],
                                       b < 0 ? -1 : B.last[b][d], cell_sum, mlo[d], mhi[d]);
        };
        region_vectors<SOUND>(B, n, f, row, r_lo, r_up, a_lo, a_up);
    }
}

// Factors of every distinct image (impact_desc.h) and block, one thread each:
// tab[(first + c) * (count + 1) + 1 + b], dimension d's items from `first`.
struct RegionItems {
    int64_t first[IMPACT_MAX_DIM + 1];
};

template <bool SOUND>
__global__ void __launch_bounds__(128)
region_items(const ImpactDesc *__restrict__ Dp, RegionItems I, RegionBoxes B, bool cell_sum,
             double2 *__restrict__ tab)
{
    const ImpactDesc &D = *Dp;
    const int slots = B.count + 1;
    const int64_t total = I.first[D.n] * slots;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t it = i / slots;
        const int b = (int)(i - it * slots) - 1;
        int d = 0;
        while (it >= I.first[d + 1]) ++d;
        int idx[IMPACT_MAX_DIM], j = 0;
        const int64_t c = it - I.first[d];
        if (D.kind != KIND_IMAGES) decode_item(D, d, c, idx, j);
        double mlo, mhi;
        image_dim<SOUND>(D, c, idx, j, d, mlo, mhi);
        const ImpactDim &g = D.dim[d];
        tab[i] = block_factor<SOUND>(g, D.edges + g.edge_off, b < 0 ? -1 : B.first[b][d],
                                     b < 0 ? -1 : B.last[b][d], cell_sum, mlo, mhi);
    }
}

// One thread per row: products of its items' factors.
template <bool SOUND>
__global__ void __launch_bounds__(256)
region_products(const ImpactDesc *__restrict__ Dp, int64_t rows, RegionItems I, RegionBoxes B,
                const double2 *__restrict__ tab, double *__restrict__ r_lo,
                double *__restrict__ r_up, double *__restrict__ a_lo, double *__restrict__ a_up)
{
    const ImpactDesc &D = *Dp;
    const int n = D.n, slots = B.count + 1;
    for (int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; row < rows;
         row += (int64_t)gridDim.x * blockDim.x) {
        int idx[IMPACT_MAX_DIM];
        int j;
        decode_row(D, row, idx, j);
        const double2 *at[IMPACT_MAX_DIM];
#pragma unroll
        for (int d = 0; d < IMPACT_MAX_DIM; ++d)
            if (d < n) at[d] = tab + (I.first[d] + item_of(D, row, idx, j, d)) * slots + 1;
        auto f = [&](int b, int d) { return at[d][b]; };
        region_vectors<SOUND>(B, n, f, row, r_lo, r_up, a_lo, a_up);
    }
}

// ---------------------------------------------------------------------------
// sampled noise: Monte-Carlo integration of the cell masses (Sec. 4.1)
// ---------------------------------------------------------------------------

constexpr int kMcThreads = 256;
constexpr int kMcThr = IMPACT_MC_EDGES_MAX + 1;   // thresholds per (row, dimension, end)

// Per-call tables: the draws' keys (dimension-major, like the draws), the
// per-dimension least and largest draw, the values u / S for every count u
// (FP64, and FP32 rounded down / up) and a flag for non-finite draws.
__global__ void __launch_bounds__(kMcThreads)
mc_prep(const double *__restrict__ samples, int n, int64_t S, long long *__restrict__ keys,
        double *__restrict__ val, float *__restrict__ val_dn, float *__restrict__ val_up,
        unsigned *__restrict__ bad)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)n * S;
         i += stride) {
        const double w = samples[i];
        if (!isfinite(w)) atomicOr(bad, 1u);
        keys[i] = dkey(w);
    }
    const double dS = (double)S;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u <= S; u += stride) {
        const double v = (double)u / dS;
        val[u] = v;
        val_dn[u] = __double2float_rd(v);
        val_up[u] = __double2float_ru(v);
    }
}

// Per-dimension least and largest draw: range[2d], range[2d + 1].
__global__ void __launch_bounds__(kMcThreads)
mc_range(const double *__restrict__ samples, int64_t S, double *__restrict__ range)
{
    __shared__ double smin[kMcThreads], smax[kMcThreads];
    const int d = blockIdx.x;
    double a = INFINITY, b = -INFINITY;
    for (int64_t s = threadIdx.x; s < S; s += blockDim.x) {
        const double w = samples[(int64_t)d * S + s];
        a = fmin(a, w);
        b = fmax(b, w);
    }
    smin[threadIdx.x] = a;
    smax[threadIdx.x] = b;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if ((int)threadIdx.x < k) {
            smin[threadIdx.x] = fmin(smin[threadIdx.x], smin[threadIdx.x + k]);
            smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[threadIdx.x + k]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        range[2 * d] = smin[0];
        range[2 * d + 1] = smax[0];
    }
}

struct McRow {
    double mlo[IMPACT_MAX_DIM], mhi[IMPACT_MAX_DIM];
    int o[IMPACT_MAX_DIM], e[IMPACT_MAX_DIM];   // window: first cell and extent per dimension
    int ws[IMPACT_MAX_DIM];                      // window strides (C order)
    int H;                                       // window cells (0: the draws all leave)
    unsigned sink_lo, sink_up;
    unsigned long long kept, dropped;
    int scan[kMcThreads / 32];
    // keys of the thresholds of edges o .. o + e, for the low and the high
    // end of the image: the draw's cell is o - 1 + #{k: key(w) >= thr[k]}
    long long thr_lo[IMPACT_MAX_DIM][kMcThr], thr_hi[IMPACT_MAX_DIM][kMcThr];
};

// #{k < cnt: t[k] <= key}, t ascending (binary search).
__device__ __forceinline__ int count_le(const long long *t, int cnt, long long key)
{
    int lo = 0, hi = cnt;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (t[mid] <= key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// One block per row (grid-stride over the rows). The draws move the row's
// image box; a block-wide histogram in shared memory counts, for every cell
// of the row's window, the draws whose moved box meets it (hu) and lies in it
// (hl). The cell of a moved end is found by integer comparisons of the draw's
// key with per-row thresholds (the FP64 decision of the definition, made
// exactly once per row and edge). The count pass writes the row's kept count,
// sink and dropped mass; the emit pass repeats the histogram and writes the
// kept cells in ascending order (cutoff 0 keeps every cell of the grid, as the
// dense definition does).
template <bool EMIT>
__global__ void __launch_bounds__(kMcThreads)
mc_rows(const ImpactDesc *__restrict__ Dp, int64_t rows, const long long *__restrict__ keys,
        int64_t S, const double *__restrict__ range, const double *__restrict__ val,
        const float *__restrict__ val_dn, const float *__restrict__ val_up, unsigned kmin,
        int hist_cap, RowOutputs o)
{
    extern __shared__ __align__(16) unsigned char mc_smem[];
    __shared__ McRow R;
    unsigned *hu = reinterpret_cast<unsigned *>(mc_smem);
    unsigned *hl = hu + hist_cap;
    const ImpactDesc &D = *Dp;
    const int n = D.n;
    const double dS = (double)S;
    const bool dense = D.cutoff <= 0.0;   // cutoff 0: every cell is kept
    const int64_t T = D.cells;
    if (EMIT && o.capacity >= 0 && o.row_ptr[o.total_at] > o.capacity) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(o.status, IMPACT_STATUS_CAPACITY);
        return;
    }
    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
        // the row's image and window: one thread per dimension
        if (threadIdx.x < (unsigned)n) {
            const int d = threadIdx.x;
            int idx[IMPACT_MAX_DIM];
            int j;
            decode_row(D, row, idx, j);
            double lo, hi;
            image_dim<false>(D, row, idx, j, d, lo, hi);
            const double mlo = fmin(lo, hi), mhi = fmax(lo, hi);   // ordered ends
            R.mlo[d] = mlo;
            R.mhi[d] = mhi;
            const ImpactDim &g = D.dim[d];
            const double *E = D.edges + g.edge_off;
            const int a = max(cell_of(E, g.N, g.inv_h, range[2 * d] + mlo), 0);
            const int b = min(cell_of(E, g.N, g.inv_h, range[2 * d + 1] + mhi), g.N - 1);
            R.o[d] = a;
            R.e[d] = b >= a ? b - a + 1 : 0;
        }
        __syncthreads();
        // the thresholds of every (dimension, edge, end), one per thread
        for (int q = threadIdx.x; q < n * 2 * kMcThr; q += blockDim.x) {
            const int d = q / (2 * kMcThr), r = q - d * (2 * kMcThr);
            const int end = r / kMcThr, k = r - end * kMcThr;
            const int ext = R.e[d];
            if (ext == 0 || ext > IMPACT_MC_EDGES_MAX || k > ext) continue;
            const ImpactDim &g = D.dim[d];
            const int edge = R.o[d] + k;
            const bool gt = edge == g.N;   // beyond the last edge: leaves the domain
            const long long t = dkey(threshold_of(end ? R.mhi[d] : R.mlo[d],
                                                  D.edges[g.edge_off + edge], gt));
            if (end) R.thr_hi[d][k] = t; else R.thr_lo[d][k] = t;
        }
        if (threadIdx.x == 0) {
            int64_t Hw = 1;
            bool wide = false;
            for (int d = 0; d < n; ++d) {
                Hw *= R.e[d];   // at most the grid's cell count
                wide = wide || R.e[d] > IMPACT_MC_EDGES_MAX;
            }
            int H = Hw < (int64_t)hist_cap ? (int)Hw : hist_cap;
            if (Hw > hist_cap || wide) {
                atomicOr(o.status, IMPACT_STATUS_MC_WINDOW);
                H = -1;
            }
            int st = 1;
            for (int d = n - 1; d >= 0; --d) {
                R.ws[d] = st;
                st *= R.e[d] > 0 ? R.e[d] : 1;
            }
            R.H = H;
            R.sink_lo = 0;
            R.sink_up = 0;
            R.kept = 0;
            R.dropped = 0;
        }
        __syncthreads();
        const int H = R.H;
        if (H < 0) {   // window too large: counted as empty, the call fails
            if (!EMIT && threadIdx.x == 0) o.row_ptr[row] = 0;
            __syncthreads();
            continue;
        }
        for (int h = threadIdx.x; h < H; h += blockDim.x) {
            hu[h] = 0;
            hl[h] = 0;
        }
        __syncthreads();
        unsigned my_sl = 0, my_su = 0;
        if (H > 0)
            for (int64_t s = threadIdx.x; s < S; s += blockDim.x) {
                // per dimension: the cells of the moved ends (integer
                // comparisons with the row's thresholds), the met range
                // relative to the window, and whether it spans two cells
                bool inside = true, outside = false, single = true, wide = false;
                int hb = 0, m2 = 0;
                unsigned pk = 0;   // dims whose met range spans two cells, 3 bits each
                int A[IMPACT_MAX_DIM], Bd[IMPACT_MAX_DIM];
#pragma unroll
                for (int d = 0; d < IMPACT_MAX_DIM; ++d) {
                    if (d < n) {
                        const long long kw = keys[(int64_t)d * S + s];
                        const int ext = R.e[d], N = D.dim[d].N;
                        const int a = R.o[d] - 1 + count_le(R.thr_lo[d], ext + 1, kw);
                        const int b = R.o[d] - 1 + count_le(R.thr_hi[d], ext + 1, kw);
                        inside = inside && a >= 0 && b <= N - 1;
                        outside = outside || b < 0 || a > N - 1;
                        single = single && a == b;
                        // relative to the window (inside it by construction;
                        // the clamps only bound malformed input)
                        const int top = ext - 1;
                        const int ad = min(max(max(a, 0) - R.o[d], 0), top);
                        const int bd = min(max(min(b, N - 1) - R.o[d], ad), top);
                        A[d] = ad;
                        Bd[d] = bd;
                        hb += ad * R.ws[d];
                        if (bd - ad == 1) {
                            pk |= (unsigned)d << (3 * m2);
                            ++m2;
                        } else if (bd - ad > 1) {
                            wide = true;
                        }
                    }
                }
                my_su += inside ? 0u : 1u;
                if (outside) {
                    ++my_sl;
                    continue;
                }
                if (single) atomicAdd(&hl[hb], 1u);
                atomicAdd(&hu[hb], 1u);
                if (!wide) {
                    // the other cells of a box of 2^m2 cells, in Gray-code
                    // order: one stride added or taken away per cell
                    int h = hb;
                    unsigned gray = 0;
                    for (unsigned k = 1; k < (1u << m2); ++k) {
                        const int j = __ffs(k) - 1;
                        const int dim = (pk >> (3 * j)) & 7;
                        const unsigned bit = 1u << j;
                        h += (gray & bit) ? -R.ws[dim] : R.ws[dim];
                        gray ^= bit;
                        atomicAdd(&hu[h], 1u);
                    }
                } else {
                    // a range of three or more cells somewhere: odometer walk
                    int c[IMPACT_MAX_DIM];
                    for (int d = 0; d < n; ++d) c[d] = A[d];
                    int h = hb;
                    while (true) {
                        int d = n - 1;
                        while (d >= 0 && c[d] == Bd[d]) {
                            h -= (c[d] - A[d]) * R.ws[d];
                            c[d] = A[d];
                            --d;
                        }
                        if (d < 0) break;
                        ++c[d];
                        h += R.ws[d];
                        atomicAdd(&hu[h], 1u);
                    }
                }
            }
        else   // every draw leaves the domain whole
            for (int64_t s = threadIdx.x; s < S; s += blockDim.x) {
                ++my_sl;
                ++my_su;
            }
        // block totals: a warp reduction, then one shared atomic per warp
        // (all threads on one shared word would serialise)
        my_sl = __reduce_add_sync(0xffffffffu, my_sl);
        my_su = __reduce_add_sync(0xffffffffu, my_su);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&R.sink_lo, my_sl);
            atomicAdd(&R.sink_up, my_su);
        }
        __syncthreads();

        if (!EMIT) {
            unsigned kept = 0;
            unsigned long long dropped = 0;
            if (!dense) {
                for (int h = threadIdx.x; h < H; h += blockDim.x) {
                    const unsigned u = hu[h];
                    if (u >= kmin) ++kept; else dropped += u;
                }
                kept = __reduce_add_sync(0xffffffffu, kept);
#pragma unroll
                for (int off = 16; off > 0; off >>= 1)
                    dropped += __shfl_xor_sync(0xffffffffu, dropped, off);
                if ((threadIdx.x & 31) == 0) {
                    atomicAdd(&R.kept, (unsigned long long)kept);
                    atomicAdd(&R.dropped, dropped);
                }
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                o.row_ptr[row] = dense ? T : (int64_t)R.kept;
                o.sink_lo[row] = (double)R.sink_lo / dS;
                o.sink_up[row] = (double)R.sink_up / dS;
                o.trunc[row] = (double)R.dropped / dS;
                if (o.flags) o.flags[row] = 0u;
            }
        } else {
            const int64_t base = o.row_ptr[row], end = o.row_ptr[row + 1];
            const bool f64 = D.prec == PREC_FP64_PLAIN;
            auto put = [&](int64_t pos, int64_t t, unsigned u, unsigned l) {
                o.col[pos] = (int32_t)t;
                if (f64) {
                    ((double *)o.up)[pos] = val[u];
                    ((double *)o.lo)[pos] = val[l];
                } else {
                    ((float *)o.up)[pos] = val_up[u];
                    ((float *)o.lo)[pos] = val_dn[l];
                }
            };
            if (dense) {
                // every cell of the grid, in order; outside the window the counts are 0
                for (int64_t t = threadIdx.x; t < T; t += blockDim.x) {
                    int64_t rest = t;
                    int h = 0;
                    bool in = H > 0;
                    for (int d = n - 1; d >= 0; --d) {
                        const int N = D.dim[d].N;
                        const int i = (int)(rest % N) - R.o[d];
                        rest /= N;
                        in = in && i >= 0 && i < R.e[d];
                        h += i * R.ws[d];
                    }
                    if (base + t < end) put(base + t, t, in ? hu[h] : 0u, in ? hl[h] : 0u);
                }
            } else {
                // the kept cells of the window in C order (ascending cell ids)
                const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
                int64_t at = 0;
                for (int h0 = 0; h0 < H; h0 += blockDim.x) {
                    const int h = h0 + threadIdx.x;
                    const bool keep = h < H && hu[h] >= kmin;
                    const unsigned m = __ballot_sync(0xffffffffu, keep);
                    if (lane == 0) R.scan[wid] = __popc(m);
                    __syncthreads();
                    int before = 0, total = 0;
                    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
                        if (k < wid) before += R.scan[k];
                        total += R.scan[k];
                    }
                    if (keep) {
                        int64_t t = 0;
                        int rest = h;
                        for (int d = 0; d < n; ++d) {
                            const int i = rest / R.ws[d];
                            rest -= i * R.ws[d];
                            t += (int64_t)(i + R.o[d]) * D.dim[d].stride;
                        }
                        const int64_t pos =
                            base + at + before + __popc(m & ((1u << lane) - 1u));
                        if (pos < end) put(pos, t, hu[h], hl[h]);
                    }
                    at += total;
                    __syncthreads();
                }
            }
        }
        __syncthreads();
    }
}

int grid_for(const void *kernel, int64_t rows)
{
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kThreads, 0);
    if (occ < 1) occ = 1;
    int64_t want = (rows + kWarpsPerBlock - 1) / kWarpsPerBlock;
    int64_t cap = (int64_t)sms * occ;
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    return (int)want;
}

}  // namespace

namespace impact {

cudaError_t launch_rows(const ImpactDesc *d_desc, int prec, bool emit, int64_t row_begin,
                        int64_t row_end, const RowOutputs &o, cudaStream_t stream)
{
    int64_t rows = row_end - row_begin;
    if (rows <= 0) return cudaSuccess;
    if (prec != PREC_FP64_PLAIN) return cudaErrorInvalidValue;
    {
        if (emit) {
            int g = grid_for((const void *)rows_fp64<true>, rows);
            rows_fp64<true><<<g, kThreads, 0, stream>>>(
                d_desc, row_begin, row_end, o.row_ptr, o.col, (double *)o.lo, (double *)o.up,
                o.sink_lo, o.sink_up, o.trunc, o.flags, o.status, o.capacity, o.total_at);
        } else {
            int g = grid_for((const void *)rows_fp64<false>, rows);
            rows_fp64<false><<<g, kThreads, 0, stream>>>(
                d_desc, row_begin, row_end, o.row_ptr, o.col, (double *)o.lo, (double *)o.up,
                o.sink_lo, o.sink_up, o.trunc, o.flags, o.status, o.capacity, o.total_at);
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_labels(const RegionBoxes &boxes, int64_t total_cells, uint8_t *labels,
                          cudaStream_t stream)
{
    if (total_cells <= 0) return cudaSuccess;
    const int64_t g = std::min<int64_t>((total_cells + 255) / 256, 152 * 16);
    label_cells<<<(unsigned)g, 256, 0, stream>>>(boxes, total_cells, labels);
    return cudaGetLastError();
}

// Items only where rows share them: below two rows per item the table's
// write and read back cost about what they save. FP64 erfc per row, dimension
// and cell bounded the per-row kernel: the 11^5 room's cell sums (1.45M rows,
// 22k items) took 50.7 ms and take 0.32 ms. Tables beyond a fixed size (it holds
// a million items of 16 boxes) are not made either: the rows need no scratch.
constexpr int64_t kRegionItemsMax = (int64_t)256 << 20;

int64_t region_scratch(const ImpactDesc &D, const RegionBoxes &boxes)
{
    int64_t items = 0;
    for (int d = 0; d < D.n; ++d) items += D.dim[d].n_items;
    const int64_t bytes = items * (boxes.count + 1) * (int64_t)sizeof(double2);
    return items <= D.rows * D.n / 2 && bytes <= kRegionItemsMax ? bytes : 0;
}

cudaError_t launch_regions(const ImpactDesc &D, const ImpactDesc *d_desc, int64_t rows,
                           const RegionBoxes &boxes, bool cell_sum, bool sound, void *scratch,
                           double *r_lo, double *r_up, double *a_lo, double *a_up,
                           cudaStream_t stream)
{
    if (rows <= 0) return cudaSuccess;
    if (scratch) {
        RegionItems I;
        I.first[0] = 0;
        for (int d = 0; d < D.n; ++d) I.first[d + 1] = I.first[d] + D.dim[d].n_items;
        for (int d = D.n; d < IMPACT_MAX_DIM; ++d) I.first[d + 1] = I.first[d];
        double2 *tab = (double2 *)scratch;
        const int64_t total = I.first[D.n] * (boxes.count + 1);
        const unsigned gi = (unsigned)std::min<int64_t>((total + 127) / 128, 152 * 64);
        const unsigned gr = (unsigned)std::min<int64_t>((rows + 255) / 256, 152 * 64);
        if (sound) {
            region_items<true><<<gi, 128, 0, stream>>>(d_desc, I, boxes, cell_sum, tab);
            region_products<true><<<gr, 256, 0, stream>>>(d_desc, rows, I, boxes, tab, r_lo, r_up,
                                                          a_lo, a_up);
        } else {
            region_items<false><<<gi, 128, 0, stream>>>(d_desc, I, boxes, cell_sum, tab);
            region_products<false><<<gr, 256, 0, stream>>>(d_desc, rows, I, boxes, tab, r_lo, r_up,
                                                           a_lo, a_up);
        }
        return cudaGetLastError();
    }
    const int64_t g = std::min<int64_t>((rows + 127) / 128, 152 * 32);
    if (sound)
        region_rows<true><<<(unsigned)g, 128, 0, stream>>>(d_desc, rows, boxes, cell_sum, r_lo,
                                                           r_up, a_lo, a_up);
    else
        region_rows<false><<<(unsigned)g, 128, 0, stream>>>(d_desc, rows, boxes, cell_sum, r_lo,
                                                            r_up, a_lo, a_up);
    return cudaGetLastError();
}

cudaError_t launch_mc_prep(const double *samples, int n, int64_t S, long long *keys,
                           double *val, float *val_dn, float *val_up, unsigned *bad,
                           double *range, cudaStream_t stream)
{
    const int64_t items = std::max<int64_t>((int64_t)n * S, S + 1);
    const int64_t g = std::min<int64_t>((items + kMcThreads - 1) / kMcThreads, 152 * 16);
    mc_prep<<<(unsigned)g, kMcThreads, 0, stream>>>(samples, n, S, keys, val, val_dn, val_up,
                                                     bad);
    mc_range<<<n, kMcThreads, 0, stream>>>(samples, S, range);
    return cudaGetLastError();
}

cudaError_t launch_mc_rows(const ImpactDesc *d_desc, bool emit, int64_t rows,
                           const long long *keys, int64_t S, const double *range,
                           const double *val, const float *val_dn, const float *val_up,
                           unsigned kmin, const RowOutputs &o, cudaStream_t stream)
{
    if (rows <= 0) return cudaSuccess;
    const int cap = IMPACT_MC_HIST_MAX;
    const size_t smem = (size_t)cap * 2 * sizeof(unsigned);
    const void *k = emit ? (const void *)mc_rows<true> : (const void *)mc_rows<false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kMcThreads, smem);
    const int64_t g = std::min<int64_t>(rows, (int64_t)sms * std::max(occ, 1));
    if (emit)
        mc_rows<true><<<(unsigned)g, kMcThreads, smem, stream>>>(
            d_desc, rows, keys, S, range, val, val_dn, val_up, kmin, cap, o);
    else
        mc_rows<false><<<(unsigned)g, kMcThreads, smem, stream>>>(
            d_desc, rows, keys, S, range, val, val_dn, val_up, kmin, cap, o);
    return cudaGetLastError();
}

int64_t scan_scratch_elems(int64_t n)
{
    return (n + kScanTile - 1) / kScanTile + 1;
}

ScanHead scan_head(int64_t *row_ptr, int64_t n, int64_t *scratch, int64_t *also)
{
    ScanHead S;
    S.row_ptr = row_ptr;
    S.tsum = scratch;
    S.also = also;
    S.n = n;
    const int64_t nt = (n + kScanTile - 1) / kScanTile;
    S.tiles = nt >= 1 && nt <= kScanHead ? (int)nt : 0;
    return S;
}

cudaError_t launch_scan(int64_t *row_ptr, int64_t n, int64_t *scratch, cudaStream_t stream,
                        int64_t *also, bool begun)
{
    const int64_t nt = std::max<int64_t>((n + kScanTile - 1) / kScanTile, 1);
    if (begun && nt == 1) return cudaSuccess;
    if (!begun && nt > 1)
        scan_tiles<<<(unsigned)nt, kScanThreads, 0, stream>>>(row_ptr, n, scratch);
    if (nt <= kScanSelf) {
        scan_apply<true><<<(unsigned)nt, kScanThreads, 0, stream>>>(row_ptr, n, scratch, also);
    } else {
        scan_sums<<<1, kScanThreads, 0, stream>>>(scratch, nt);
        scan_apply<false><<<(unsigned)nt, kScanThreads, 0, stream>>>(row_ptr, n, scratch, also);
    }
    return cudaGetLastError();
}

}  // namespace impact
