// synth.cu -- interval-iteration controller synthesis on a device-resident
// IMDP (impact_synthesize / impact_synthesize_ex, include/impact.h): the
// paper's Alg. 3 (safety) and Alg. 4 (reach-avoid), pessimistic or optimistic
// policy (Sec. 5), infinite or finite horizon (Remark 5.1), the disturbance
// points as an adversary, with the linear program of Sec. 5 solved per row by
// the sorting method of Sec. 6.2.
//
// Per row the successors are the kept target cells t with [lo_t, up_t], the
// out-of-domain sink with [sink_lo, sink_up] and the truncated mass as one
// more successor with [0, trunc]; with region vectors (Sec. 3.1) the
// labelled cells and the sink give way to the target region [R_min, R_max]
// and the avoid region [A_min, A_max]. The sorting method starts every successor
// at its lower bound and raises them in ascending (min LP) or descending (max
// LP) order of their value until the total is 1. Instead of sorting a row, one
// warp finds the value threshold tau of that greedy fill: with w = up - lo and
// G(x) = sum of w over the successors whose value is <= x, tau is the least x
// with G(x) >= 1 - sum lo. Every row compares the same value vector, so each
// iteration ranks the cells once (sort of their order-preserving keys, equal
// values share a rank) and a row bisects over ranks, log2(cells) steps of
// 32-bit compares and exact integer sums. The remaining mass is valued just
// below tau when the result must not be too high (the V0 update of a min LP)
// and at tau otherwise, so V0 stays below and V1 above their exact values.
// The max LP is the min LP of the values 1 - v.
//
// One warp per row computes the row's LP for both vectors; one thread per cell
// then keeps the best input (or the policy's) and writes the cell's next V0
// and V1; the largest |V1 - V0| is gathered with an atomic max on the bits of
// a non-negative double. The stopping test runs on the device: launches go out
// a few iterations ahead of the host's look at it, and those past the last
// iteration return at once.
//
// What bounds it: the row kernel's FP64 multiplies and adds (2 lanes per clock
// and SM on this part), about five per successor and vector; their order is
// part of the result (ties between inputs), so it is kept. Dense robot 21x21
// (3969 rows of 441 successors, about 270 iterations): 44 -> 16 ms; a 62-step
// bisection over the doubles for each vector took 140 us of an iteration's 200,
// the host's stopping test 50. Now 37 for the rows, 6 for the cells, 4 for the
// ranks.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "../../include/impact.h"
#include "alloc.h"
#include "plan.h"

namespace {

constexpr int kThreads = 256;
constexpr int kRowThreads = 128;
constexpr int kCache = 16;    // successors per lane kept in registers (rows <= 512)

#define CK(expr)                                                                              \
    do {                                                                                      \
        cudaError_t e_ = (expr);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return impact::fail(e_ == cudaErrorMemoryAllocation ? IMPACT_ERR_OOM              \
                                                                : IMPACT_ERR_CUDA,            \
                                std::string(#expr) + ": " + cudaGetErrorString(e_));          \
    } while (0)

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of a value per vector over the warp: the lower half-warp gets V0's sum,
// the upper V1's, each the bits of warp_sum (the same tree of additions). Five
// adds and not ten: the FP64 pipe is busy as long with one active lane as with
// 32, so the halves work side by side.
__device__ __forceinline__ double half_sum(double v0, double v1, int lane)
{
    const unsigned m = 0xffffffffu;
    double x = lane & 16 ? v1 : v0;
    x += __shfl_xor_sync(m, lane & 16 ? v0 : v1, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(m, x, o);
    return x;
}

// The same for two values per vector (a, b): six adds and not twenty.
__device__ __forceinline__ void half_sums(const double (&a)[2], const double (&b)[2], int lane,
                                          double &sa, double &sb)
{
    const unsigned m = 0xffffffffu;
    const bool up = lane & 16, right = lane & 8;
    double x = up ? a[1] : a[0], y = up ? b[1] : b[0];
    x += __shfl_xor_sync(m, up ? a[0] : a[1], 16);
    y += __shfl_xor_sync(m, up ? b[0] : b[1], 16);
    double s = right ? y : x;
    s += __shfl_xor_sync(m, right ? x : y, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(m, s, o);
    const double other = __shfl_xor_sync(m, s, 8);
    sa = right ? other : s;
    sb = right ? s : other;
}

// Order-preserving integer key of a finite double (-0 and +0 share key 0):
// x <= y exactly when okey(x) <= okey(y).
__device__ __forceinline__ long long okey(double x)
{
    const long long b = __double_as_longlong(x);
    if ((b & 0x7fffffffffffffffll) == 0) return 0;   // +0 and -0, without an FP64 compare
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffll);
}

// The double whose key is k (the inverse of okey; key -1 gives -0).
__device__ __forceinline__ double from_okey(long long k)
{
    return __longlong_as_double(k >= 0 ? k : (k ^ 0x7fffffffffffffffll));
}

// What the rows read of the cells, both vectors side by side: the values as the
// min LP sees them (max LP: 1 - v), and their ranks (0 is the value 0's, one
// past every smaller key a cell's; two 16-bit halves when they fit).
struct Seen {
    const double2 *val;            // [cells]
    const int2 *rank;              // [cells], or
    const unsigned *packed;        // [cells] V0's rank below, V1's above
    const long long *key[2];       // [cells + 2] key of a rank
    const int *one;                // [2] the rank of the value 1
};

template <bool PACKED>
__device__ __forceinline__ int2 ranks_at(const Seen &Q, int32_t t)
{
    if (!PACKED) return Q.rank[t];
    const unsigned p = Q.packed[t];
    return make_int2((int)(p & 0xffffu), (int)(p >> 16));
}

// Iteration state on the device.
struct Step {
    unsigned long long diff;   // bits of max |V1 - V0| of the running iteration
    int done, its;             // stopping test met; iterations finished
};

struct RowRef {
    int64_t a, b;           // successor range in col/lo/up
    // three further successors: the sink and an empty one, or the two regions;
    // then the truncated mass. Bounds, widths, and whether the min LP sees them
    // with value 1 (else 0)
    double xlo[3], xw[3];
    bool one[3];
    double rest;            // 1 - sum of all lower bounds
};

// Mass the lower bounds of a row leave and widths of its further successors,
// in 2^-52 units.
struct RowFix {
    long long rest, xw[3];
};

// Sum over the warp of 64-bit integers: three 32-bit warp sums of 27-bit pieces.
__device__ __forceinline__ long long warp_sum_ll(long long x)
{
    const unsigned m = 0xffffffffu, k = (1u << 27) - 1u;
    const unsigned lo = __reduce_add_sync(m, (unsigned)x & k);
    const unsigned mid = __reduce_add_sync(m, (unsigned)(x >> 27) & k);
    const int hi = __reduce_add_sync(m, (int)(x >> 54));
    return (long long)lo + ((long long)mid << 27) + ((long long)hi << 54);
}

// Greedy (sorting-method) optimum of one row for both value vectors at once:
// for V0 (the remaining mass valued low) in the lower half-warp, for V1 (valued
// high) in the upper.
// `excl`: when not null, successors t with excl[t] != 0 are left out (their
// mass is in the region successors). Short rows (SHORT: at most 512) load their
// successors in unrolled, independent steps and keep ranks and widths in
// registers for the whole bisection; long rows read them again in every pass.
template <typename VT, bool PACKED, bool SHORT>
__device__ __forceinline__ double row_lp(const RowRef &R, const RowFix &F,
                                         const int32_t *__restrict__ col,
                                         const VT *__restrict__ lo, const VT *__restrict__ up,
                                         const long long *__restrict__ wfix,
                                         const uint8_t *__restrict__ excl, const Seen &Q,
                                         bool maximize)
{
    constexpr int kKeep = SHORT ? kCache : 1;
    const int lane = threadIdx.x & 31;
    auto out = [&](int32_t t) { return excl != nullptr && excl[t] != 0; };
    const int len = (int)min(R.b - R.a, (int64_t)INT_MAX);
    double slov[2] = {0.0, 0.0};
    int rank0[kKeep], rank1[kKeep];     // SHORT
    unsigned pair[kKeep];               // SHORT and PACKED
    long long w[kKeep];
    auto lower = [&](double l, double2 v) {
        slov[0] += l * v.x;
        slov[1] += l * v.y;
    };
    if (SHORT) {
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            const int i = lane + 32 * k;
            rank0[k] = rank1[k] = INT_MAX;
            pair[k] = 0xffffffffu;
            w[k] = 0;
            if (i < len) {
                const int32_t t = col[R.a + i];
                if (!out(t)) {
                    if (PACKED) {
                        pair[k] = Q.packed[t];
                    } else {
                        const int2 r = Q.rank[t];
                        rank0[k] = r.x;
                        rank1[k] = r.y;
                    }
                    w[k] = wfix[R.a + i];
                    lower((double)lo[R.a + i], Q.val[t]);
                }
            }
        }
    } else {
        for (int64_t i = R.a + lane; i < R.b; i += 32) {
            const int32_t t = col[i];
            if (!out(t)) lower((double)lo[i], Q.val[t]);
        }
    }
    double sum = half_sum(slov[0], slov[1], lane);
#pragma unroll
    for (int x = 0; x < 3; ++x)
        if (R.one[x]) sum += R.xlo[x];
    if (R.rest <= 0.0) return maximize ? 1.0 - sum : sum;
    // G over ranks: mass (2^-52 units) of the successors of rank <= m
    long long base = 0, top = 0;   // the further successors of value 0 and 1
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (R.one[k]) top += F.xw[k]; else base += F.xw[k];
    }
    int l[2] = {-1, -1}, h[2] = {Q.one[0], Q.one[1]};
    const int one[2] = {h[0], h[1]};
    auto narrow = [&](int v, int m, long long g) {
        if (h[v] - l[v] <= 1) return;
        g += base + (m >= one[v] ? top : 0);
        if (g >= F.rest) h[v] = m; else l[v] = m;
    };
    while (h[0] - l[0] > 1 || h[1] - l[1] > 1) {
        const int m0 = l[0] + ((h[0] - l[0]) >> 1), m1 = l[1] + ((h[1] - l[1]) >> 1);
        long long g0 = 0, g1 = 0;
        if (SHORT) {
            const unsigned s1 = ((unsigned)m1 << 16) | 0xffffu;
#pragma unroll
            for (int k = 0; k < kKeep; ++k) {
                if (PACKED ? (int)(pair[k] & 0xffffu) <= m0 : rank0[k] <= m0) g0 += w[k];
                if (PACKED ? pair[k] <= s1 : rank1[k] <= m1) g1 += w[k];
            }
        } else {
            for (int64_t i = R.a + lane; i < R.b; i += 32) {
                const int32_t t = col[i];
                if (out(t)) continue;
                const int2 r = ranks_at<PACKED>(Q, t);
                const long long x = wfix[i];
                if (r.x <= m0) g0 += x;
                if (r.y <= m1) g1 += x;
            }
        }
        narrow(0, m0, warp_sum_ll(g0));
        narrow(1, m1, warp_sum_ll(g1));
    }
    // the mass below tau and its weighted value, in FP64 (nothing is below
    // when no mass is left to place)
    const int cut0 = F.rest > 0 ? h[0] : 0, cut1 = F.rest > 0 ? h[1] : 0;
    double g[2] = {0.0, 0.0}, gv[2] = {0.0, 0.0};
    auto below = [&](int64_t i, bool b0, bool b1) {
        if (!(b0 || b1)) return;
        const double x = (double)up[i] - (double)lo[i];
        const double2 v = Q.val[col[i]];
        if (b0) {
            g[0] += x;
            gv[0] += x * v.x;
        }
        if (b1) {
            g[1] += x;
            gv[1] += x * v.y;
        }
    };
    if (SHORT) {
        const unsigned s1 = (unsigned)cut1 << 16;
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            const bool b0 = PACKED ? (int)(pair[k] & 0xffffu) < cut0 : rank0[k] < cut0;
            const bool b1 = PACKED ? pair[k] < s1 : rank1[k] < cut1;
            below(R.a + lane + 32 * k, b0, b1);
        }
    } else {
        for (int64_t i = R.a + lane; i < R.b; i += 32) {
            const int32_t t = col[i];
            if (out(t)) continue;
            const int2 r = ranks_at<PACKED>(Q, t);
            below(i, r.x < cut0, r.y < cut1);
        }
    }
    double below_w, below_v;
    half_sums(g, gv, lane, below_w, below_v);
    // tau and the double before it; the further successors of value 0 lie
    // below it when it is positive (those of value 1 never do)
    const bool high = lane & 16;
    const long long kh = F.rest > 0 ? (high ? Q.key[1][h[1]] : Q.key[0][h[0]]) : okey(-1.0) + 1;
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (!R.one[k] && kh > 0) below_w += R.xw[k];
    const double x = from_okey(maximize == high ? kh - 1 : kh);
    const double y = sum + below_v + (R.rest - below_w) * fmax(x, 0.0);
    return maximize ? 1.0 - y : y;
}

struct Phase {
    int spec;         // IMPACT_REACH_AVOID or IMPACT_SAFETY
    bool choose;      // optimise over the inputs (phase 1) or follow the policy
    bool maximize;    // the LP direction
    bool pol_v1;      // phase 1: the policy follows the V1 choice (else V0)
    int n_disturb;    // disturbance points per input
};

// Region vectors of the rows (all four, or all null).
struct Regions {
    const double *r_lo, *r_up, *a_lo, *a_up;
};

// The further successors of row r: the regions or the sink, then the truncated
// mass at its worst end (0 in a min LP, 1 in a max LP).
__device__ __forceinline__ void further(const Phase &ph, const Regions &rg, int64_t r,
                                        const double *__restrict__ sink_lo,
                                        const double *__restrict__ sink_up,
                                        const double *__restrict__ trunc, RowRef &R)
{
    const bool reach = ph.spec == IMPACT_REACH_AVOID;
    bool one[3];   // the successor's value, before the max LP's v -> 1 - v
    if (rg.r_lo) {
        // the target region (reach: value 1) and the avoid region with the
        // sink (safety: value 1)
        R.xlo[0] = rg.r_lo[r];
        R.xw[0] = rg.r_up[r] - rg.r_lo[r];
        one[0] = reach;
        R.xlo[1] = rg.a_lo[r];
        R.xw[1] = rg.a_up[r] - rg.a_lo[r];
        one[1] = !reach;
    } else {
        R.xlo[0] = sink_lo[r];
        R.xw[0] = sink_up[r] - sink_lo[r];
        one[0] = !reach;
        R.xlo[1] = 0.0;
        R.xw[1] = 0.0;
        one[1] = false;
    }
    R.xlo[2] = 0.0;
    R.xw[2] = trunc[r];
    one[2] = ph.maximize;
#pragma unroll
    for (int k = 0; k < 3; ++k) R.one[k] = one[k] != ph.maximize;
}

// What no iteration changes: per pair the width up - lo in 2^-52 units (the
// bisection sums integers), per row the mass the lower bounds leave.
template <typename VT>
__global__ void __launch_bounds__(kThreads)
row_prep(Phase ph, int64_t rows, int64_t per_cell, const uint8_t *__restrict__ labels,
         const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
         const VT *__restrict__ lo, const VT *__restrict__ up, const double *__restrict__ sink_lo,
         const double *__restrict__ sink_up, const double *__restrict__ trunc, Regions rg,
         long long *__restrict__ wfix, double *__restrict__ rest, RowFix *__restrict__ fix)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = warp0; r < rows; r += nwarps) {
        if (labels[r / per_cell] != 0) continue;   // absorbing: its rows are never used
        RowRef R;
        further(ph, rg, r, sink_lo, sink_up, trunc, R);
        double slo = 0.0;
        for (int64_t i = row_ptr[r] + lane; i < row_ptr[r + 1]; i += 32) {
            const double l = (double)lo[i];
            wfix[i] = __double2ll_rn(((double)up[i] - l) * 0x1p52);
            if (!rg.r_lo || labels[col[i]] == 0) slo += l;
        }
        slo = warp_sum(slo);
#pragma unroll
        for (int x = 0; x < 3; ++x) slo += R.xlo[x];
        if (lane == 0) {
            const double left = 1.0 - slo;
            rest[r] = left;
            RowFix f;
            f.rest = __double2ll_rn(left * 0x1p52);
#pragma unroll
            for (int x = 0; x < 3; ++x) f.xw[x] = __double2ll_rn(R.xw[x] * 0x1p52);
            fix[r] = f;
        }
    }
}

// The LP of every row the phase needs (all inputs in phase 1, the policy's in
// phase 2), one warp per row, for both vectors: V0 never rises above, V1 never
// falls below the exact update.
template <typename VT, bool PACKED>
__global__ void __launch_bounds__(kRowThreads)
row_values(Phase ph, const Step *__restrict__ step, int64_t rows, int n_inputs,
           const uint8_t *__restrict__ labels, const int64_t *__restrict__ row_ptr,
           const int32_t *__restrict__ col, const VT *__restrict__ lo, const VT *__restrict__ up,
           const double *__restrict__ sink_lo, const double *__restrict__ sink_up,
           const double *__restrict__ trunc, const long long *__restrict__ wfix,
           const double *__restrict__ rest, const RowFix *__restrict__ fix, Regions rg, Seen Q,
           const int32_t *__restrict__ policy, double *__restrict__ R0, double *__restrict__ R1)
{
    if (step->done) return;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t per_cell = (int64_t)n_inputs * ph.n_disturb;
    const uint8_t *excl = rg.r_lo ? labels : nullptr;
    for (int64_t r = warp0; r < rows; r += nwarps) {
        const int64_t c = r / per_cell;
        const int j = (int)((r - c * per_cell) / ph.n_disturb);
        if (labels[c] != 0 || (!ph.choose && j != policy[c])) continue;
        RowRef R;
        R.a = row_ptr[r];
        R.b = row_ptr[r + 1];
        R.rest = rest[r];
        further(ph, rg, r, sink_lo, sink_up, trunc, R);
        const RowFix F = fix[r];
        const double res =
            R.b - R.a <= 32 * kCache
                ? row_lp<VT, PACKED, true>(R, F, col, lo, up, wfix, excl, Q, ph.maximize)
                : row_lp<VT, PACKED, false>(R, F, col, lo, up, wfix, excl, Q, ph.maximize);
        if (lane == 0) R0[r] = res;
        if (lane == 16) R1[r] = res;
    }
}

// The disturbance's choice among the W rows of one input: the least
// satisfaction (reach-avoid) or the most unsafe value (safety).
__device__ __forceinline__ double worst(const double *__restrict__ p, int W, bool reach)
{
    double w = p[0];
    for (int k = 1; k < W; ++k) w = reach ? fmin(w, p[k]) : fmax(w, p[k]);
    return w;
}

// Cell c: for each input the disturbance's worst row, then the best input
// (phase 1) or the policy's input (phase 2): the next V0 and V1. The values are
// satisfaction probabilities (reach-avoid: inputs maximise, disturbances
// minimise) or unsafe ones (safety: inputs minimise, disturbances maximise).
__device__ __forceinline__ void cell_next(const Phase &ph, int64_t c, int n_inputs,
                                          const uint8_t *__restrict__ labels,
                                          const double *__restrict__ R0,
                                          const double *__restrict__ R1,
                                          int32_t *__restrict__ policy, double &n0, double &n1)
{
    const bool reach = ph.spec == IMPACT_REACH_AVOID;
    const int W = ph.n_disturb;
    const uint8_t lab = labels[c];
    if (lab != 0) {   // absorbing: target (reach) or avoid (safety) has value 1
        n0 = n1 = (reach ? lab == 1 : lab == 2) ? 1.0 : 0.0;
        if (ph.choose) policy[c] = 0;
    } else if (ph.choose) {
        double b0 = 0.0, b1 = 0.0;
        int arg0 = 0, arg1 = 0;
#pragma unroll 4
        for (int j = 0; j < n_inputs; ++j) {
            const double a = worst(R0 + (c * n_inputs + j) * W, W, reach);
            const double b = worst(R1 + (c * n_inputs + j) * W, W, reach);
            if (j == 0 || (reach ? a > b0 : a < b0)) {
                b0 = a;
                arg0 = j;
            }
            if (j == 0 || (reach ? b > b1 : b < b1)) {
                b1 = b;
                arg1 = j;
            }
        }
        policy[c] = ph.pol_v1 ? arg1 : arg0;
        n0 = b0;
        n1 = b1;
    } else {
        n0 = worst(R0 + (c * n_inputs + policy[c]) * W, W, reach);
        n1 = worst(R1 + (c * n_inputs + policy[c]) * W, W, reach);
    }
    n0 = fmin(fmax(n0, 0.0), 1.0);
    n1 = fmin(fmax(n1, 0.0), 1.0);
}

// V0 from 0 and V1 from 1 on the free cells (from 0 both, for a finite
// horizon); the labelled cells hold their absorbing value.
__device__ __forceinline__ void cell_start(const Phase &ph, bool horizon, uint8_t lab, double &a,
                                           double &b)
{
    const bool reach = ph.spec == IMPACT_REACH_AVOID;
    if (lab == 0) {
        a = 0.0;
        b = horizon ? 0.0 : 1.0;
    } else {
        a = b = (reach ? lab == 1 : lab == 2) ? 1.0 : 0.0;
    }
}

// The stopping test of Alg. 3/4 (eps < 0: none, a finite horizon).
__device__ __forceinline__ void end_step(Step *step, double diff, double eps)
{
    step->its += 1;
    if (eps >= 0.0 && diff <= eps) step->done = 1;
}

// Least index of sorted[0..n) whose key is not below x.
__device__ __forceinline__ int lower_bound(const long long *sorted, int n, long long x)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (sorted[mid] < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Rank of a key among the cells' sorted keys: 0 is the value 0's; equal keys
// share one.
__device__ __forceinline__ int rank_of(const long long *sorted, int n, long long key)
{
    return key == 0 ? 0 : 1 + lower_bound(sorted, n, key);
}

// The cells' values of one step, and what the rows read of them (struct Seen).
struct Cells {
    double *V0, *V1;
    long long *keys;       // [2][cells]
    double2 *val;
    int2 *rank;
    unsigned *packed;
    long long *key[2];
    int *one;
};

// The next (FIRST: the start) values, as seen by the rows, and their keys, one
// thread per cell.
template <bool FIRST>
__global__ void __launch_bounds__(kThreads)
cell_update(Phase ph, bool horizon, Step *__restrict__ step, int64_t cells, int n_inputs,
            const uint8_t *__restrict__ labels, const double *__restrict__ R0,
            const double *__restrict__ R1, Cells C, int32_t *__restrict__ policy)
{
    if (!FIRST && step->done) return;
    double dmax = 0.0;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < cells;
         c += (int64_t)gridDim.x * blockDim.x) {
        double a, b;
        if (FIRST) cell_start(ph, horizon, labels[c], a, b);
        else cell_next(ph, c, n_inputs, labels, R0, R1, policy, a, b);
        C.V0[c] = a;
        C.V1[c] = b;
        dmax = fmax(dmax, fabs(b - a));
        if (ph.maximize) {
            a = 1.0 - a;
            b = 1.0 - b;
        }
        C.val[c] = make_double2(a, b);
        C.keys[c] = okey(a);
        C.keys[cells + c] = okey(b);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (!FIRST && (threadIdx.x & 31) == 0 && dmax > 0.0)
        atomicMax(&step->diff, (unsigned long long)__double_as_longlong(dmax));
}

// Stores the ranks of a cell; the thread of cell 0 also those of the values 0
// and 1.
__device__ __forceinline__ void put_ranks(const Cells &C, bool packed, int64_t c, int r0, int r1,
                                          long long k0, long long k1)
{
    if (packed) C.packed[c] = (unsigned)r0 | ((unsigned)r1 << 16);
    else C.rank[c] = make_int2(r0, r1);
    C.key[0][r0] = k0;
    C.key[1][r1] = k1;
}
__device__ __forceinline__ void put_ends(const Cells &C, int v, int one)
{
    C.one[v] = one;
    C.key[v][0] = 0;
    C.key[v][one] = okey(1.0);
}

// Few cells: ranks by counting the smaller keys, one warp per cell, and the
// stopping test by block 0 (a block that finds the step already ended has
// nothing left to rank for). Work cells^2: below 4096 cells it takes a few
// microseconds over the whole chip, where a sort in one block takes twenty.
constexpr int kCountCells = 4096;

__global__ void __launch_bounds__(kThreads)
rank_count(Step *step, bool first, double eps, int cells, bool packed, Cells C)
{
    if (step->done) return;
    const int lane = threadIdx.x & 31;
    const int warp0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int c = warp0; c <= cells; c += nwarps) {   // c == cells: the value 1
        const long long k0 = c < cells ? C.keys[c] : okey(1.0);
        const long long k1 = c < cells ? C.keys[cells + c] : okey(1.0);
        int r0 = 0, r1 = 0;
        for (int i = lane; i < cells; i += 32) {
            r0 += C.keys[i] < k0;
            r1 += C.keys[cells + i] < k1;
        }
        r0 = k0 == 0 ? 0 : 1 + __reduce_add_sync(0xffffffffu, r0);
        r1 = k1 == 0 ? 0 : 1 + __reduce_add_sync(0xffffffffu, r1);
        if (lane == 0) {
            if (c < cells) {
                put_ranks(C, packed, c, r0, r1, k0, k1);
            } else {
                put_ends(C, 0, r0);
                put_ends(C, 1, r1);
            }
        }
    }
    if (!first && blockIdx.x == 0 && threadIdx.x == 0) {
        end_step(step, __longlong_as_double((long long)step->diff), eps);
        step->diff = 0;
    }
}

// Sort of both vectors' keys: tiles in shared memory, then merge passes in
// which every element finds its place in the neighbouring run.
constexpr int kTile = 2048;
constexpr int kBlockThreads = 1024;

__global__ void __launch_bounds__(kBlockThreads)
sort_tiles(const Step *__restrict__ step, int64_t cells, const long long *__restrict__ keys,
           long long *__restrict__ sorted)
{
    __shared__ long long key[kTile];
    if (step->done) return;
    const int64_t base = (int64_t)blockIdx.x * kTile, at = blockIdx.y * cells;
    for (int i = threadIdx.x; i < kTile; i += blockDim.x)
        key[i] = base + i < cells ? keys[at + base + i] : LLONG_MAX;
    __syncthreads();
    for (int k = 2; k <= kTile; k <<= 1)
        for (int s = k >> 1; s > 0; s >>= 1) {
            for (int q = threadIdx.x; q < kTile / 2; q += blockDim.x) {
                const int i = ((q / s) * 2 * s) + (q % s);
                const long long u = key[i], w = key[i + s];
                if ((u > w) == ((i & k) == 0)) {
                    key[i] = w;
                    key[i + s] = u;
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < kTile; i += blockDim.x)
        if (base + i < cells) sorted[at + base + i] = key[i];
}

__global__ void __launch_bounds__(kThreads)
merge_runs(const Step *__restrict__ step, int64_t cells, int64_t run,
           const long long *__restrict__ in, long long *__restrict__ out)
{
    if (step->done) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 2 * cells;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = i >= cells, c = i - v * cells;
        const long long *x = in + v * cells;
        const int64_t pair = c / (2 * run) * (2 * run);
        const int64_t mid = min(pair + run, cells), end = min(pair + 2 * run, cells);
        const long long k = x[c];
        // the first run's elements go before equal ones of the second
        int64_t lo = c < mid ? mid : pair, hi = c < mid ? end : mid;
        const int64_t from = lo;
        while (lo < hi) {
            const int64_t m = (lo + hi) >> 1;
            if (c < mid ? x[m] < k : x[m] <= k) lo = m + 1; else hi = m;
        }
        out[v * cells + (c < mid ? c : pair + (c - mid)) + (lo - from)] = k;
    }
}

// Ranks from the sorted keys.
__global__ void __launch_bounds__(kThreads)
rank_cells(const Step *__restrict__ step, int64_t cells, bool packed,
           const long long *__restrict__ sorted, Cells C)
{
    if (step->done) return;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < cells;
         c += (int64_t)gridDim.x * blockDim.x) {
        const long long k0 = C.keys[c], k1 = C.keys[cells + c];
        put_ranks(C, packed, c, rank_of(sorted, (int)cells, k0),
                  rank_of(sorted + cells, (int)cells, k1), k0, k1);
        if (c == 0) {
            put_ends(C, 0, rank_of(sorted, (int)cells, okey(1.0)));
            put_ends(C, 1, rank_of(sorted + cells, (int)cells, okey(1.0)));
        }
    }
}

__global__ void step_end(Step *step, double eps)
{
    if (step->done) return;
    end_step(step, __longlong_as_double((long long)step->diff), eps);
    step->diff = 0;
}

__global__ void __launch_bounds__(kThreads)
finish(int spec, int64_t cells, const double *__restrict__ V, bool complement,
       double *__restrict__ out)
{
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < cells;
         c += (int64_t)gridDim.x * blockDim.x)
        out[c] = complement ? 1.0 - V[c] : V[c];
}

int grid_of(int64_t items, int per_block)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (items + per_block - 1) / per_block;
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * 8));
}

bool device_array(const void *p)
{
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" impact_status impact_synthesize_ex(const impact_csr *imdp, impact_precision precision,
                                              int64_t cells, int n_inputs, const uint8_t *labels,
                                              const impact_synth_options *opt, double *p_min,
                                              double *p_max, int32_t *policy, int *iterations,
                                              void *stream)
{
    using impact::fail;
    if (!imdp || !opt) return fail(IMPACT_ERR_ARG, "null IMDP or options");
    if (precision != IMPACT_FP32_SOUND && precision != IMPACT_FP64_PLAIN)
        return fail(IMPACT_ERR_ARG, "unknown precision");
    const int spec = opt->spec;
    if (spec != IMPACT_REACH_AVOID && spec != IMPACT_SAFETY)
        return fail(IMPACT_ERR_ARG, "unknown specification");
    if (opt->optimistic != 0 && opt->optimistic != 1)
        return fail(IMPACT_ERR_ARG, "optimistic must be 0 or 1");
    if (opt->horizon < 0) return fail(IMPACT_ERR_ARG, "horizon must be >= 0");
    const int W = opt->n_disturb;
    if (W < 1) return fail(IMPACT_ERR_ARG, "n_disturb must be >= 1");
    if (cells < 1 || n_inputs < 1 || imdp->rows != cells * n_inputs * W)
        return fail(IMPACT_ERR_ARG, "the IMDP must have cells * n_inputs * n_disturb rows");
    const bool horizon = opt->horizon > 0;
    if (!horizon && (!(opt->eps > 0.0) || opt->max_iters < 1))
        return fail(IMPACT_ERR_ARG, "eps > 0 and max_iters >= 1");
    if (!device_array(imdp->row_ptr) || !device_array(imdp->sink_lo) ||
        !device_array(imdp->sink_up) || !device_array(imdp->trunc) || !device_array(labels) ||
        !device_array(p_min) || !device_array(p_max) || !device_array(policy) ||
        (imdp->nnz > 0 && (!device_array(imdp->col) || !device_array(imdp->lo) ||
                           !device_array(imdp->up))))
        return fail(IMPACT_ERR_ARG, "the IMDP, labels and outputs must be device arrays");
    Regions rg{opt->r_lo, opt->r_up, opt->a_lo, opt->a_up};
    const int given = !!rg.r_lo + !!rg.r_up + !!rg.a_lo + !!rg.a_up;
    if (given != 0 && given != 4) return fail(IMPACT_ERR_ARG, "give all four region vectors or none");
    if (given == 4 && (!device_array(rg.r_lo) || !device_array(rg.r_up) ||
                       !device_array(rg.a_lo) || !device_array(rg.a_up)))
        return fail(IMPACT_ERR_ARG, "the region vectors must be device arrays");
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t rows = imdp->rows;
    const int64_t nnz = imdp->nnz;
    const bool count = cells <= kCountCells;   // ranks by counting (else by sorting)
    const bool packed = cells + 2 <= 0xffff;   // a rank fits 16 bits
    double *buf = nullptr, *rbuf = nullptr;
    long long *kbuf = nullptr, *wfix = nullptr;
    double2 *vbuf = nullptr;
    int *ibuf = nullptr;
    Step *d_step = nullptr, *h_step = nullptr;
    cudaEvent_t seen[2] = {nullptr, nullptr};
    auto free_all = [&]() {
        impact::dev_free_async(buf, st);
        impact::dev_free_async(kbuf, st);
        impact::dev_free_async(vbuf, st);
        impact::dev_free_async(ibuf, st);
        impact::dev_free_async(wfix, st);
        impact::dev_free_async(rbuf, st);
        impact::dev_free_async(d_step, st);
        cudaStreamSynchronize(st);
        impact::host_free(h_step);
        for (cudaEvent_t e : seen)
            if (e) cudaEventDestroy(e);
    };
    {
        // V0, V1 and their next values; what the rows see of them; keys of
        // the cells, of a rank and, for the sort, two buffers; per-row values
        // and remaining mass
        cudaError_t e = impact::dev_malloc_async(&buf, (size_t)cells * 4 * sizeof(double), st);
        if (e == cudaSuccess)
            e = impact::dev_malloc_async(&vbuf, (size_t)cells * sizeof(double2), st);
        if (e == cudaSuccess)
            e = impact::dev_malloc_async(
                &kbuf, (size_t)(2 * cells + 2 * (cells + 2) + (count ? 0 : 4 * cells)) *
                           sizeof(long long), st);
        if (e == cudaSuccess)
            e = impact::dev_malloc_async(&ibuf, (size_t)(2 * cells + 2) * sizeof(int), st);
        if (e == cudaSuccess)
            e = impact::dev_malloc_async(
                &wfix, (size_t)std::max<int64_t>(nnz, 1) * sizeof(long long), st);
        if (e == cudaSuccess)
            e = impact::dev_malloc_async(&rbuf, (size_t)rows * (3 * sizeof(double) + sizeof(RowFix)),
                                         st);
        if (e == cudaSuccess) e = impact::dev_malloc_async(&d_step, sizeof(Step), st);
        if (e == cudaSuccess) e = impact::host_malloc(&h_step, 2 * sizeof(Step));
        for (cudaEvent_t &x : seen)
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&x, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            free_all();
            return fail(e == cudaErrorMemoryAllocation ? IMPACT_ERR_OOM : IMPACT_ERR_CUDA,
                        std::string("synthesis scratch: ") + cudaGetErrorString(e));
        }
    }
    const bool reach = spec == IMPACT_REACH_AVOID;
    // the LP that bounds satisfaction from below: reach-avoid the min LP,
    // safety the max LP of the unsafe value; phase 1 optimises the inputs on
    // it (pessimistic) or on the other one (optimistic)
    const bool lower_max = !reach;
    const bool lp1_max = opt->optimistic ? !lower_max : lower_max;
    const int limit = horizon ? opt->horizon : opt->max_iters;
    const double eps = horizon ? -1.0 : opt->eps;
    const int g_cells = grid_of(cells, kThreads);
    const int g_rows = grid_of(rows, kThreads / 32);
    const int g_lp = grid_of(rows, kRowThreads / 32);
    impact_status status = IMPACT_OK;
    int its[2] = {0, 0};
    RowFix *fix = (RowFix *)rbuf;
    double *R0 = (double *)(fix + rows), *R1 = R0 + rows, *rest = R1 + rows;
    const float *lo32 = (const float *)imdp->lo, *up32 = (const float *)imdp->up;
    const double *lo64 = (const double *)imdp->lo, *up64 = (const double *)imdp->up;
    const bool f32 = precision == IMPACT_FP32_SOUND;
    for (int phase = 0; phase < 2 && status == IMPACT_OK; ++phase) {
        Phase ph;
        ph.spec = spec;
        ph.choose = phase == 0;
        ph.maximize = phase == 0 ? lp1_max : !lp1_max;
        // the vector whose end phase 1 reports: reach min LP -> V0, reach max
        // LP -> V1, safety max LP -> V1 (P_min = 1 - V1), min LP -> V0
        ph.pol_v1 = lp1_max;
        ph.n_disturb = W;
        if (phase == 0) {
            const int64_t per_cell = (int64_t)n_inputs * W;
            if (f32)
                row_prep<float><<<g_rows, kThreads, 0, st>>>(
                    ph, rows, per_cell, labels, imdp->row_ptr, imdp->col, lo32, up32,
                    imdp->sink_lo, imdp->sink_up, imdp->trunc, rg, wfix, rest, fix);
            else
                row_prep<double><<<g_rows, kThreads, 0, st>>>(
                    ph, rows, per_cell, labels, imdp->row_ptr, imdp->col, lo64, up64,
                    imdp->sink_lo, imdp->sink_up, imdp->trunc, rg, wfix, rest, fix);
        }
        // the values of step i are in half i & 1; the rest is of the latest
        auto cells_of = [&](int i) {
            Cells C;
            C.V0 = buf + 2 * (i & 1) * cells;
            C.V1 = C.V0 + cells;
            C.keys = kbuf;
            C.val = vbuf;
            C.rank = (int2 *)ibuf;
            C.packed = (unsigned *)ibuf;
            C.key[0] = kbuf + 2 * cells;
            C.key[1] = C.key[0] + cells + 2;
            C.one = ibuf + 2 * cells;
            return C;
        };
        auto rank_all = [&](int i, bool first) {   // keys -> ranks, and the stopping test
            const Cells C = cells_of(i);
            if (count) {
                rank_count<<<grid_of(cells + 1, kThreads / 32), kThreads, 0, st>>>(
                    d_step, first, eps, (int)cells, packed, C);
                return;
            }
            long long *in = C.key[1] + cells + 2, *out = in + 2 * cells;
            const dim3 tiles((unsigned)((cells + kTile - 1) / kTile), 2);
            sort_tiles<<<tiles, kBlockThreads, 0, st>>>(d_step, cells, C.keys, in);
            for (int64_t run = kTile; run < cells; run *= 2) {
                merge_runs<<<grid_of(2 * cells, kThreads), kThreads, 0, st>>>(d_step, cells, run,
                                                                             in, out);
                std::swap(in, out);
            }
            rank_cells<<<g_cells, kThreads, 0, st>>>(d_step, cells, packed, in, C);
            if (!first) step_end<<<1, 1, 0, st>>>(d_step, eps);
        };
        auto start = [&]() {
            cudaMemsetAsync(d_step, 0, sizeof(Step), st);
            cell_update<true><<<g_cells, kThreads, 0, st>>>(ph, horizon, d_step, cells, n_inputs,
                                                            labels, R0, R1, cells_of(0), policy);
            rank_all(0, true);
        };
        const Cells C0 = cells_of(0);
        const Seen Q{C0.val, C0.rank, C0.packed, {C0.key[0], C0.key[1]}, C0.one};
        auto rows_step = [&](auto kernel, auto *lo, auto *up) {
            kernel<<<g_lp, kRowThreads, 0, st>>>(ph, d_step, rows, n_inputs, labels, imdp->row_ptr,
                                                 imdp->col, lo, up, imdp->sink_lo, imdp->sink_up,
                                                 imdp->trunc, wfix, rest, fix, rg, Q, policy, R0, R1);
        };
        auto iterate = [&](int i) {   // values of step i -> those of step i + 1
            if (f32 && packed) rows_step(row_values<float, true>, lo32, up32);
            else if (f32) rows_step(row_values<float, false>, lo32, up32);
            else if (packed) rows_step(row_values<double, true>, lo64, up64);
            else rows_step(row_values<double, false>, lo64, up64);
            cell_update<false><<<g_cells, kThreads, 0, st>>>(ph, horizon, d_step, cells, n_inputs,
                                                             labels, R0, R1, cells_of(i + 1),
                                                             policy);
            rank_all(i + 1, false);
        };
        start();
        // launches go out in groups; the host looks at a group's outcome when
        // the next one is queued, so the device does not wait for it
        constexpr int kAhead = 8;
        int sent = 0, group = 0;
        bool done = false;
        while (!done && status == IMPACT_OK) {
            const int to = std::min(limit, sent + kAhead);
            const bool fresh = to > sent;
            for (; sent < to; ++sent) iterate(sent);
            cudaError_t e = cudaGetLastError();
            if (e == cudaSuccess && fresh) {
                e = cudaMemcpyAsync(h_step + (group & 1), d_step, sizeof(Step),
                                    cudaMemcpyDeviceToHost, st);
                if (e == cudaSuccess) e = cudaEventRecord(seen[group & 1], st);
                ++group;
            }
            // the group before this one, or the last one when nothing is left
            const int look = fresh && sent < limit ? group - 2 : group - 1;
            if (e == cudaSuccess && look >= 0) {
                e = cudaEventSynchronize(seen[look & 1]);
                done = h_step[look & 1].done != 0 || h_step[look & 1].its >= limit;
                its[phase] = h_step[look & 1].its;
            }
            if (e != cudaSuccess) status = fail(IMPACT_ERR_CUDA, cudaGetErrorString(e));
        }
        if (status != IMPACT_OK) break;
        // reach-avoid: the min LP gives P_min = V0, the max LP P_max = V1;
        // safety: the max LP gives P_min = 1 - V1, the min LP P_max = 1 - V0
        double *dst;
        if (reach) dst = ph.maximize ? p_max : p_min;
        else dst = ph.maximize ? p_min : p_max;
        const Cells last = cells_of(its[phase]);
        const double *src = ph.maximize ? last.V1 : last.V0;
        finish<<<g_cells, kThreads, 0, st>>>(spec, cells, src, !reach, dst);
        if (horizon && cudaStreamSynchronize(st) != cudaSuccess)
            status = fail(IMPACT_ERR_CUDA, "synthesis phase failed");
    }
    free_all();
    if (iterations) {
        iterations[0] = its[0];
        iterations[1] = its[1];
    }
    return status;
}

extern "C" impact_status impact_synthesize(const impact_csr *imdp, impact_precision precision,
                                           int64_t cells, int n_inputs, const uint8_t *labels,
                                           int spec, double eps, int max_iters, double *p_min,
                                           double *p_max, int32_t *policy, int *iterations,
                                           void *stream)
{
    impact_synth_options o;
    memset(&o, 0, sizeof(o));
    o.spec = spec;
    o.n_disturb = 1;
    o.eps = eps;
    o.max_iters = max_iters;
    return impact_synthesize_ex(imdp, precision, cells, n_inputs, labels, &o, p_min, p_max,
                                policy, iterations, stream);
}
