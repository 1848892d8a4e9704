// walk_fp32.cu -- FP32-sound construction (Def. 3.1 with outward rounding,
// Sec. 4.4 cutoff, Remark 4.1 sink).
//
//   setup       From the interval image of the source cell: the window of
//               target cells that can pass the cutoff, erf/erfc once per window
//               edge at the image's lower and upper end, and the window's factor
//               table: U[t] >= the largest Gaussian mass of target t over the
//               image (T_max of Def. 3.1 relaxed to the image box) and L[t] <= the
//               smallest (T_min), trimmed to the targets that pass on their own.
//               Rows that read the same coordinates and input offset share an
//               image (impact_desc.h): items_fp32 makes each window once and
//               rows_fp32 gathers a row's into its record; systems whose images
//               are distinct make them per row (setup_fp32, one lane per row and
//               dimension). The lanes of a row exchange their window maxima and
//               sums by shuffles for the pruning thresholds.
//   leaf_fp32   the sorted leaf tables (below) of the distinct images of the
//               last two dimensions, and their entries by kept count.
//   terms_fp32  after the count pass, one thread per row: sink bounds, mass of
//               the targets outside the window box, truncated mass and row
//               checks (FP64, outward).
//   walk_fp32   one warp per row, persistent (rows from an atomic counter in
//               ascending order). It walks the prefix tree of target cells
//               level by level in C order over the first n - 2 dimensions: a
//               node at level k is a prefix (t_0..t_k) with the RU-rounded
//               product P of its upper factors; the children of a list of
//               nodes are enumerated as candidates, one lane each, a child is
//               kept iff RU(P U[t]) can still reach the cutoff under the
//               largest factors of the later dimensions, and the warp compacts
//               the kept ones (ballot + popc) into the next level's list (lists
//               hold kCap nodes; longer expansions are taken in chunks, depth
//               first, so leaves come out in C order). The last two dimensions
//               form one leaf table per row, B[a, b] = RU(U[a] U[b]) (and the
//               RD product of the lower factors), so a pair's bound is one more
//               product RU(P B[a, b]). The count pass finds how many entries of
//               B pass under each parent by a binary search in B sorted by
//               value, with prefix sums for the row sums (B from the row's shared
//               leaf table, else sorted by the warp). The emit pass stores
//               the kept pairs warp-contiguously: from the lists of a shared
//               table of 20 to 48 entries, one lane per kept pair, else every
//               entry of B tested under each parent, one lane each.
//
// Kernel modes: COUNT (pairs per row, truncated mass, row checks), EMIT
// (pairs at given row offsets) and FUSED (both: each row publishes its pair
// count, finds its offset by a decoupled look-back over the rows before it,
// and writes its pairs).
//
// Upper bounds are products rounded up, lower bounds products rounded down,
// associated as ((..(U_0 U_1) ..) U_{n-3}) (U_{n-2} U_{n-1}) whatever the
// enumeration order, so a pair's value depends only on its row. Every
// lane-to-candidate assignment is a function of the row alone, so per-lane
// partial sums and their fixed reduction tree give the same bits under every
// launch shape and in every batch.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <limits.h>

#include <algorithm>

#include "../../include/impact.h"
#include "impact_desc.h"
#include "kernels.h"
#include "launch.h"
#include "rowmath.cuh"
#include "scan.cuh"
#include "sound_fp32.cuh"

namespace {

using rowmath::fastdiv;
using rowmath::find_problem;

constexpr float kTwoM44 = 5.6843419e-14f;       // 2^-44
constexpr float kGrow18 = 1.0000038147f;        // 1 + 2^-18

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// (sh, sl) += p, exactly in sh (TwoSum) with the rounding error kept in sl.
__device__ __forceinline__ void acc_pair(float &sh, float &sl, float2 p)
{
    float s = __fadd_rn(sh, p.x);
    float bb = __fsub_rn(s, sh);
    float e = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bb)), __fsub_rn(p.x, bb));
    sh = s;
    sl = __fadd_rn(sl, __fadd_rn(e, p.y));
}

// (rh, rl) = a - (bh, bl)
__device__ __forceinline__ void sub_pair(float2 a, float bh, float bl, float &rh, float &rl)
{
    float s = __fsub_rn(a.x, bh);
    float bb = __fsub_rn(s, a.x);
    float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bb)), __fsub_rn(-bh, bb));
    rh = s;
    rl = __fadd_rn(__fsub_rn(a.y, bl), e);
}

__device__ __forceinline__ float fpred(float x) { return nextafterf(x, 0.0f); }
__device__ __forceinline__ float fsucc(float x) { return nextafterf(x, INFINITY); }

// Smallest float y with RU(y * r) >= c (c > 0 a float, r >= 0): RU(y r) >= c
// iff y r > pred(c), and the smallest float above pred(c)/r is
// succ(RD(pred(c)/r)) whether or not that quotient is a float.
__device__ __forceinline__ float threshold(float c, float r)
{
    if (!(r > 0.0f)) return INFINITY;
    return fsucc(__fdiv_rd(fpred(c), r));
}

// Edge point: alpha = (E - m)/(sigma sqrt2) at one image end, its half-width
// and its tails.
struct EdgePt {
    float a, da;
    sound::TailPair t;
};

// The target midpoint lies at or below / at or above the mean, certainly.
__device__ __forceinline__ bool mid_below(const EdgePt &c, const EdgePt &e)
{
    return __fadd_ru(__fadd_ru(c.a, c.da), __fadd_ru(e.a, e.da)) <= 0.0f;
}
__device__ __forceinline__ bool mid_above(const EdgePt &c, const EdgePt &e)
{
    return __fadd_rd(__fsub_rd(c.a, c.da), __fsub_rd(e.a, e.da)) >= 0.0f;
}

// One dimension of a row: the window [a, a + W) of target cells that can
// pass the cutoff and, in erf units, rho = (E_a - m)/(sigma sqrt2) at both
// image ends as FP32 pairs (edge a + k is then rho + k kappa).
struct Win {
    int a, W;
    float kh, kl, err;          // kappa (cell width in erf units) pair, edge error
    float rh0, rl0, rh1, rl1;   // rho at m_lo and m_hi, pairs
};

__device__ __forceinline__ EdgePt edge_at(const Win &h, int k, bool hi_end)
{
    EdgePt e;
    sound::alpha_point(k, h.kh, h.kl, h.err, hi_end ? h.rh1 : h.rh0, hi_end ? h.rl1 : h.rl0, e.a,
                       e.da);
    e.t = sound::tails(e.a, e.da);
    return e;
}

// The interval image of the source cell in dimension d (affine sign
// split or unicycle trig ranges from host tables, or the caller's images),
// the window [a, a + W) of targets that can pass the cutoff (every target
// outside lies more than delta beyond the image), and rho = (E_a - m) /
// (sigma sqrt2) at both image ends as FP32 pairs. False if the window
// exceeds the planner's bound wcap.
__device__ bool dim_window(const ImpactDesc &D, int64_t row, const int *idx, int j, int d, Win &h)
{
    const int n = D.n;
    int my_idx = 0, idx2 = idx[2 < IMPACT_MAX_DIM ? 2 : 0];
#pragma unroll
    for (int k = 0; k < IMPACT_MAX_DIM; ++k)
        if (k == d) my_idx = idx[k];
    const ImpactDim &g = D.dim[d];

    float mulo = 0.0f, muhi = 0.0f;   // image ends in cells (window placement only)
    float m0h = 0.0f, m0l = 0.0f, m1h = 0.0f, m1l = 0.0f, mag = 0.0f;
    double dmlo = 0.0, dmhi = 0.0;
    if (D.kind == KIND_AFFINE) {
#pragma unroll
        for (int k = 0; k < IMPACT_MAX_DIM; ++k) {
            if (k < n) {
                int t = (d * n + k) * D.n_max + idx[k];
                mulo += D.mu_lo[t];
                muhi += D.mu_hi[t];
                float2 pl = D.ta_lo[t], ph = D.ta_hi[t];
                acc_pair(m0h, m0l, pl);
                acc_pair(m1h, m1l, ph);
                mag += fabsf(pl.x) + fabsf(ph.x);
            }
        }
        float2 o = D.oa[j * n + d];
        acc_pair(m0h, m0l, o);
        acc_pair(m1h, m1l, o);
        mag += 2.0f * fabsf(o.x);
        float mo = D.mo[j * n + d];
        mulo += mo;
        muhi += mo;
    } else if (D.kind == KIND_UNICYCLE) {
        const float2 *ea = D.ea + g.edge_off;
        float2 xlo = ea[my_idx], xhi = ea[my_idx + 1];
        acc_pair(m0h, m0l, xlo);
        acc_pair(m1h, m1l, xhi);
        float2 vl, vh;
        float cl, ch;
        if (d == 2) {
            vl = vh = D.oma[j];
            cl = ch = D.omm[j];
        } else {
            int t = (idx2 * D.n_inputs + j) * 4 + 2 * d;
            vl = D.ua[t];
            vh = D.ua[t + 1];
            cl = D.um[t];
            ch = D.um[t + 1];
        }
        acc_pair(m0h, m0l, vl);
        acc_pair(m1h, m1l, vh);
        mag += fabsf(xlo.x) + fabsf(xhi.x) + fabsf(vl.x) + fabsf(vh.x);
        mulo = (float)my_idx + cl;
        muhi = (float)(my_idx + 1) + ch;
    } else {
        const double *im = D.images + (row * n + d) * 2;
        dmlo = im[0];
        dmhi = im[1];
        mulo = (float)((dmlo - g.lo) * g.inv_h);
        muhi = (float)((dmhi - g.lo) * g.inv_h);
    }
    // conservative window [a, a + W): every target outside has U below the
    // cutoff (its cell lies more than delta beyond the image)
    const float dc = g.delta_cells;
    float xa = floorf(mulo - dc - 1e-3f - 1e-5f * fabsf(mulo));
    float xb = floorf(muhi + dc + 1e-3f + 1e-5f * fabsf(muhi));
    const float top = (float)(g.N - 1);
    xa = fminf(fmaxf(xa, 0.0f), top);
    xb = fminf(fmaxf(xb, 0.0f), top);
    const int a = (int)xa;
    const int W = max((int)xb - a + 1, 1);
    h.a = a;
    h.W = W;
    if (W > g.wcap) return false;
    float2 ea = D.ea[g.edge_off + a];
    if (D.kind == KIND_IMAGES) {
        const double Ea = D.edges[g.edge_off + a];
        sound::split_pair((Ea - dmlo) * g.inv_s, h.rh0, h.rl0);
        sound::split_pair((Ea - dmhi) * g.inv_s, h.rh1, h.rl1);
        mag = (float)((fabs(Ea) + fabs(dmlo) + fabs(dmhi)) * g.inv_s);
    } else {
        sub_pair(ea, m0h, m0l, h.rh0, h.rl0);
        sub_pair(ea, m1h, m1l, h.rh1, h.rl1);
        mag += fabsf(ea.x);
    }
    h.kh = g.kappa_hi;
    h.kl = g.kappa_lo;
    h.err = __fadd_ru(g.edge_err, __fmul_ru(__fmul_ru(mag, 4.0f), kTwoM44));
    return true;
}


// ---------------------------------------------------------------------------
// setup: one record per row
// ---------------------------------------------------------------------------

// Per (row, dimension) entry of a row record. The record is RecDim[n], RecRow,
// then the window tables, (U, L) pairs, dimension d's at entry rec_off[d].
struct RecDim {
    int tw;          // trimmed width: targets first..last that pass on their own
    int tb;          // table entry of the first trimmed target
    int cb;          // column of the first trimmed target: (a + first) * stride
    uint32_t magic;  // ceil(2^32 / tw) when tw > 1: e / tw = umulhi(e, magic)
    float cp;        // least child product whose subtree can still reach the cutoff
    float SR;        // RU product of the later dimensions' window sums
    int stride;      // column stride of the dimension (C order)
    int lay;         // the walk's layout (tw <= 32): lanes hold floor(32 / tw) parents
                     // (bits 0-15), a chunk is floor(kCap / tw) whole parents of
                     // candidates (bits 16-31); wider windows: 0
};
static_assert(sizeof(RecDim) == 32, "RecDim layout");

// Per-row entry of the record, between the dimensions' entries and the tables.
struct RecRow {
    int64_t leaf;    // the row's leaf table (builds that share them)
    int64_t pad;
};

__device__ __forceinline__ RecRow *rec_row(unsigned char *rec, int n)
{
    return reinterpret_cast<RecRow *>(rec + sizeof(RecDim) * n);
}
__device__ __forceinline__ float2 *rec_table(unsigned char *rec, int n)
{
    return reinterpret_cast<float2 *>(rec + sizeof(RecDim) * n + sizeof(RecRow));
}

// Leaf table of the last two dimensions that a row with these digits shares.
__device__ __forceinline__ int64_t leaf_of_row(const ImpactDesc &D, const int *idx, int j)
{
    if (!D.leaf_shared) return 0;
    int64_t c = D.leaf_cls[j];
#pragma unroll
    for (int k = 0; k < IMPACT_MAX_DIM; ++k)
        if (k < D.n) c += (int64_t)idx[k] * D.leaf_mul[k];
    return c;
}

// Everything of one (row, dimension) that needs no other dimension.
struct DimOut {
    int tw = 0, f0 = 0, a = 0;
    float M = 0.0f;     // largest U
    float SW = 0.0f;    // sum of U over the trimmed window (rounded up)
    float O = 0.0f;     // mass outside the trimmed window (rounded up)
    float qlo = 0.0f, qhi = 0.0f;   // out-of-domain mass bounds
};
static_assert(sizeof(DimOut) == 32, "DimOut layout");

// The window of dimension d of a row and its factor table, written to `ul`
// (the record's entries of dimension d): U[k], L[k] for target a + k from the
// tails of its two edges at both image ends (neighbouring targets share an
// edge), then the trimmed window, its sums and the out-of-domain bounds.
__device__ DimOut setup_dim(const ImpactDesc &D, int64_t row, const int *idx, int j, int d,
                            float2 *ul, uint32_t *status)
{
    DimOut o;
    Win h;
    if (!dim_window(D, row, idx, j, d, h)) {
        atomicOr(status, IMPACT_STATUS_TABLE_OVERFLOW);
        return o;
    }
    const ImpactDim &g = D.dim[d];
    const float cut = D.cutoff32;
    o.a = h.a;
    EdgePt c0 = edge_at(h, 0, false), c1 = edge_at(h, 0, true);
    const EdgePt w0 = c0;   // edge a at m_lo (left tail below)
    int first = -1, last = -1;
    float pre = 0.0f, mid = 0.0f, post = 0.0f, M = 0.0f;
    for (int k = 0; k < h.W; ++k) {
        const EdgePt e0 = edge_at(h, k + 1, false), e1 = edge_at(h, k + 1, true);
        float U, L;
        if (mid_below(c0, e0)) {            // target midpoint <= m_lo
            U = sound::cell_hi(c0.a, c0.t, e0.a, e0.t);
            L = sound::cell_lo(c1.a, c1.t, e1.a, e1.t);
        } else if (mid_above(c1, e1)) {     // target midpoint >= m_hi
            U = sound::cell_hi(c1.a, c1.t, e1.a, e1.t);
            L = sound::cell_lo(c0.a, c0.t, e0.a, e0.t);
        } else {                            // midpoint may be inside
            U = g.plateau_hi;
            L = fminf(sound::cell_lo(c0.a, c0.t, e0.a, e0.t),
                      sound::cell_lo(c1.a, c1.t, e1.a, e1.t));
        }
        ul[k] = make_float2(U, L);
        if (U >= cut) {
            if (first < 0) {
                first = k;
                mid = U;
            } else {
                mid = __fadd_ru(mid, __fadd_ru(post, U));
                post = 0.0f;
            }
            last = k;
            M = fmaxf(M, U);
        } else if (first < 0) {
            pre = __fadd_ru(pre, U);
        } else {
            post = __fadd_ru(post, U);
        }
        c0 = e0;
        c1 = e1;
    }
    // c1 is now edge a + W at m_hi
    float O = __fadd_ru(pre, post);
    const EdgePt lo0 = edge_at(h, -h.a, false), hi0 = edge_at(h, g.N - h.a, false);
    const EdgePt lo1 = edge_at(h, -h.a, true), hi1 = edge_at(h, g.N - h.a, true);
    if (h.a > 0)   // cells 0..a-1 lie left of the image: their mass at m_lo
        O = __fadd_ru(O, sound::cell_hi(lo0.a, lo0.t, w0.a, w0.t));
    if (h.a + h.W < g.N)   // cells right of the window: their mass at m_hi
        O = __fadd_ru(O, sound::cell_hi(c1.a, c1.t, hi1.a, hi1.t));
    // out-of-domain mass Q(m) = T(-alpha(lo_D)) + T(alpha(hi_D))
    const float q0 = __fadd_ru(lo0.t.m_hi, hi0.t.p_hi);
    const float q1 = __fadd_ru(lo1.t.m_hi, hi1.t.p_hi);
    o.qhi = fminf(fmaxf(q0, q1), 1.0f);
    float qlo;
    if (mid_below(lo0, hi0))
        qlo = __fadd_rd(lo0.t.m_lo, hi0.t.p_lo);
    else if (mid_above(lo1, hi1))
        qlo = __fadd_rd(lo1.t.m_lo, hi1.t.p_lo);
    else
        qlo = g.qmin_lo;
    o.qlo = fminf(qlo, 1.0f);
    o.tw = first >= 0 ? last - first + 1 : 0;
    o.f0 = first >= 0 ? first : 0;
    o.M = M;
    o.SW = mid;
    o.O = O;
    return o;
}

// The pieces of setup_dim for a window that several lanes make. (setup_dim keeps
// its own text: built from these, setup_fp32 took 1.06 ms for 24 random systems,
// not 1.01.) Bounds of a target's factor from its edges c, e at the image's lower
// (0) and upper (1) end.
__device__ __forceinline__ float2 target_factor(const ImpactDim &g, const EdgePt &c0,
                                                const EdgePt &e0, const EdgePt &c1,
                                                const EdgePt &e1)
{
    if (mid_below(c0, e0))              // target midpoint <= m_lo
        return make_float2(sound::cell_hi(c0.a, c0.t, e0.a, e0.t),
                           sound::cell_lo(c1.a, c1.t, e1.a, e1.t));
    if (mid_above(c1, e1))              // target midpoint >= m_hi
        return make_float2(sound::cell_hi(c1.a, c1.t, e1.a, e1.t),
                           sound::cell_lo(c0.a, c0.t, e0.a, e0.t));
    return make_float2(g.plateau_hi,    // midpoint may be inside
                       fminf(sound::cell_lo(c0.a, c0.t, e0.a, e0.t),
                             sound::cell_lo(c1.a, c1.t, e1.a, e1.t)));
}

// The trimmed window and its sums, targets taken in order.
struct Trim {
    int first = -1, last = -1;
    float pre = 0.0f, mid = 0.0f, post = 0.0f, M = 0.0f;
    __device__ __forceinline__ void take(int k, float U, float cut)
    {
        if (U >= cut) {
            if (first < 0) {
                first = k;
                mid = U;
            } else {
                mid = __fadd_ru(mid, __fadd_ru(post, U));
                post = 0.0f;
            }
            last = k;
            M = fmaxf(M, U);
        } else if (first < 0) {
            pre = __fadd_ru(pre, U);
        } else {
            post = __fadd_ru(post, U);
        }
    }
};

// The rest of a window: the mass outside it and the out-of-domain bounds, from
// its first edge at m_lo (w0), its last at m_hi (w1) and the domain's edges.
__device__ __forceinline__ DimOut dim_out(const ImpactDim &g, const Win &h, const Trim &s,
                                          const EdgePt &w0, const EdgePt &w1, const EdgePt &lo0,
                                          const EdgePt &hi0, const EdgePt &lo1, const EdgePt &hi1)
{
    DimOut o;
    o.a = h.a;
    float O = __fadd_ru(s.pre, s.post);
    if (h.a > 0)   // cells 0..a-1 lie left of the image: their mass at m_lo
        O = __fadd_ru(O, sound::cell_hi(lo0.a, lo0.t, w0.a, w0.t));
    if (h.a + h.W < g.N)   // cells right of the window: their mass at m_hi
        O = __fadd_ru(O, sound::cell_hi(w1.a, w1.t, hi1.a, hi1.t));
    // out-of-domain mass Q(m) = T(-alpha(lo_D)) + T(alpha(hi_D))
    const float q0 = __fadd_ru(lo0.t.m_hi, hi0.t.p_hi);
    const float q1 = __fadd_ru(lo1.t.m_hi, hi1.t.p_hi);
    o.qhi = fminf(fmaxf(q0, q1), 1.0f);
    float qlo;
    if (mid_below(lo0, hi0))
        qlo = __fadd_rd(lo0.t.m_lo, hi0.t.p_lo);
    else if (mid_above(lo1, hi1))
        qlo = __fadd_rd(lo1.t.m_lo, hi1.t.p_lo);
    else
        qlo = g.qmin_lo;
    o.qlo = fminf(qlo, 1.0f);
    o.tw = s.first >= 0 ? s.last - s.first + 1 : 0;
    o.f0 = s.first >= 0 ? s.first : 0;
    o.M = s.M;
    o.SW = s.mid;
    o.O = O;
    return o;
}

// A lane's edge point seen by the others of its group of G.
template <int G>
__device__ __forceinline__ EdgePt edge_from(const EdgePt &e, int src)
{
    EdgePt r;
    r.a = __shfl_sync(0xffffffffu, e.a, src, G);
    r.da = __shfl_sync(0xffffffffu, e.da, src, G);
    r.t.p_lo = __shfl_sync(0xffffffffu, e.t.p_lo, src, G);
    r.t.p_hi = __shfl_sync(0xffffffffu, e.t.p_hi, src, G);
    r.t.m_lo = __shfl_sync(0xffffffffu, e.t.m_lo, src, G);
    r.t.m_hi = __shfl_sync(0xffffffffu, e.t.m_hi, src, G);
    return r;
}

// setup_dim by a group of G lanes (4 or 8), one edge each per round: the same
// values, all lanes of the warp together (inactive groups: act false). Few
// windows leave most of the chip idle and take as long as the longest chain of
// tails, which this cuts to the rounds; many are cheaper one lane each, since
// here every lane of a group repeats the image and the sums.
template <int G>
__device__ DimOut setup_dim_split(const ImpactDesc &D, int64_t row, const int *idx, int j, int d,
                                  float2 *ul, uint32_t *status, bool act)
{
    const int lane = threadIdx.x & (G - 1);
    Win h;
    h.W = -1;
    h.a = 0;
    if (act && !dim_window(D, row, idx, j, d, h)) {
        if (lane == 0) atomicOr(status, IMPACT_STATUS_TABLE_OVERFLOW);
        act = false;
    }
    const ImpactDim &g = D.dim[d];
    const int W = act ? h.W : -1;   // edges 0..W
    const int rounds = __reduce_max_sync(0xffffffffu, (W + G) / G);
    EdgePt x{}, y{}, last0{}, last1{};
    Trim s;
    for (int r = 0; r < rounds; ++r) {
        const int k = r * G + lane;
        x = EdgePt{};
        y = EdgePt{};
        if (k <= W) {
            x = edge_at(h, k, false);
            y = edge_at(h, k, true);
        }
        // target k - 1 lies between the edges of the lane before and this one
        EdgePt c0 = edge_from<G>(x, (lane + G - 1) & (G - 1));
        EdgePt c1 = edge_from<G>(y, (lane + G - 1) & (G - 1));
        const EdgePt n0 = edge_from<G>(x, G - 1), n1 = edge_from<G>(y, G - 1);
        if (lane == 0) {
            c0 = last0;
            c1 = last1;
        }
        last0 = n0;
        last1 = n1;
        float2 f = make_float2(0.0f, 0.0f);
        if (k >= 1 && k <= W) {
            f = target_factor(g, c0, x, c1, y);
            ul[k - 1] = f;
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const float U = __shfl_sync(0xffffffffu, f.x, i, G);
            const int kk = r * G + i;
            if (kk >= 1 && kk <= W) s.take(kk - 1, U, D.cutoff32);
        }
    }
    // the window's and the domain's edges, one lane each
    auto end = [&](int i) {
        const int k = i < 4 ? (i & 1 ? g.N : 0) - h.a : i == 4 ? 0 : h.W;
        return edge_at(h, k, i == 2 || i == 3 || i == 5);
    };
    x = EdgePt{};
    y = EdgePt{};
    if (act && lane < 6) x = end(lane);
    if (G == 4 && act && lane < 2) y = end(4 + lane);
    const EdgePt w0 = G == 4 ? edge_from<G>(y, 0) : edge_from<G>(x, 4);
    const EdgePt w1 = G == 4 ? edge_from<G>(y, 1) : edge_from<G>(x, 5);
    const EdgePt lo0 = edge_from<G>(x, 0), hi0 = edge_from<G>(x, 1);
    const EdgePt lo1 = edge_from<G>(x, 2), hi1 = edge_from<G>(x, 3);
    return act ? dim_out(g, h, s, w0, w1, lo0, hi0, lo1, hi1) : DimOut();
}

// What one lane of a row's dimensions finishes with the row's others (the
// lanes of a row are `base`, `base + step`, .. one per dimension): its record entry with the
// pruning threshold (a child t of a node with product P survives iff
// RU(RU(P U[t]) R') >= cutoff, R' the product of the later dimensions' largest
// factors grown by 2^-18 to cover the rounding of the rest of the chain; cp is
// the least such child product).
__device__ __forceinline__ void finish_dim(const ImpactDesc &D, const DimOut &o, int d, int base,
                                           bool act, unsigned char *rr, int step = 1)
{
    const int n = D.n;
    float R = 1.0f, SR = 1.0f;
#pragma unroll
    for (int k = 0; k < IMPACT_MAX_DIM; ++k) {
        if (k < n) {   // n is the same for the whole warp
            const int src = (base + k * step) & 31;
            const float Mk = __shfl_sync(0xffffffffu, o.M, src);
            const float SWk = __shfl_sync(0xffffffffu, o.SW, src);
            if (k > d) {
                R = __fmul_ru(R, Mk);
                SR = __fmul_ru(SR, SWk);
            }
        }
    }
    if (!act) return;
    const float cut = D.cutoff32;
    RecDim rd;
    rd.tw = o.tw;
    rd.tb = D.dim[d].rec_off + o.f0;
    rd.cb = (o.a + o.f0) * D.dim[d].stride;
    rd.magic = o.tw > 1 ? 0xffffffffu / (unsigned)o.tw + 1u : 0u;   // ceil(2^32 / tw)
    rd.cp = 0.0f;
    if (cut > 0.0f) rd.cp = (d == n - 1) ? cut : threshold(cut, __fmul_ru(R, kGrow18));
    rd.SR = SR;
    rd.stride = D.dim[d].stride;
    rd.lay = (o.tw >= 1 && o.tw <= 32)
                 ? ((32 / o.tw) | (((IMPACT_WALK_CAP / o.tw) * o.tw) << 16)) : 0;
    reinterpret_cast<RecDim *>(rr)[d] = rd;
}

// The numbers of one (row, dimension) that the row terms need.
__device__ __forceinline__ float4 term_of(const DimOut &o)
{
    return make_float4(o.SW, o.O, o.qlo, o.qhi);
}

// (double)x, by its bits where x is +0 or a positive normal: the conversion
// takes the FP64 pipe, which bounds the row terms (0.222 to 0.189 ms for the 11^5
// room, 0.232 to 0.193 for the 7-D building). Other values convert.
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x);
    const bool odd = b - 0x00800000u >= 0x7f000000u;
    if (__builtin_expect(odd && b != 0u, 0)) return (double)x;
    return odd ? 0.0 : __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}

// terms_fp32: the FP64 row terms, one thread per row: sink bounds and the mass
// of the targets outside the window box, with outward rounding, and after a
// count pass (acc: its FP32 sums per row: dropped mass, upper and lower bounds
// of the kept pairs) the truncated mass and the row checks of Def. 3.1.
// FP64 issues two lanes per clock and SM here, whatever share of a warp's
// lanes is active: in the setup (n lanes per row) and at the end of a row's
// walk (one lane) the same operations took 1.1 ms of the 11^5 room's 12.
constexpr int kTermThreads = 256;
__global__ void __launch_bounds__(kTermThreads)
terms_fp32(const BatchIndex *__restrict__ B, const float4 *__restrict__ acc, int64_t fault_row,
           double *__restrict__ sink_lo, double *__restrict__ sink_up, double *__restrict__ trunc,
           uint32_t *__restrict__ flags, uint32_t *__restrict__ status, impact::ScanHead scan)
{
    if (blockIdx.x < scan.tiles) {   // the row-pointer scan, in blocks of its own
        rowscan::first_pass<kTermThreads>(scan);
        return;
    }
    const int64_t rows = B->rows, step = (int64_t)(gridDim.x - scan.tiles) * kTermThreads;
    for (int64_t row = (int64_t)(blockIdx.x - scan.tiles) * kTermThreads + threadIdx.x; row < rows;
         row += step) {
        const int q = find_problem(B->row_begin, B->count, row);
        const ImpactDesc &D = *B->desc[q];
        const int n = D.n;
        const int64_t rl = row - B->row_begin[q];
        int idx[IMPACT_MAX_DIM], j = 0;
        if (D.share32) rowmath::decode_row(D, rl, idx, j);
        const float4 *own = reinterpret_cast<const float4 *>(B->terms[q]) + rl * n;
        double pin_up = 1.0, pin_dn = 1.0, out = 0.0, pre = 1.0;
#pragma unroll
        for (int k = 0; k < IMPACT_MAX_DIM; ++k) {
            if (k < n) {
                float4 v;
                if (D.share32) {
                    const ImpactDim &g = D.dim[k];
                    v = term_of(*reinterpret_cast<const DimOut *>(
                        B->items[q] + g.item_off +
                        rowmath::item_of(D, rl, idx, j, k) * g.item_stride));
                } else {
                    v = own[k];
                }
                const double SWk = widen(v.x), Ok = widen(v.y);
                // sink: 1 - prod_k (1 - Q_k)
                pin_up = __dmul_ru(pin_up, __dsub_ru(1.0, widen(v.z)));
                pin_dn = __dmul_rd(pin_dn, __dsub_rd(1.0, widen(v.w)));
                // mass outside the window box, partitioned by the first
                // dimension that leaves its window:
                // sum_k prod_{i<k} SW_i * O_k * prod_{i>k} (SW_i + O_i)
                out = __dadd_ru(__dmul_ru(out, __dadd_ru(SWk, Ok)), __dmul_ru(pre, Ok));
                pre = __dmul_ru(pre, SWk);
            }
        }
        const double sl = fmax(__dsub_rd(1.0, pin_up), 0.0), su = fmin(__dsub_ru(1.0, pin_dn), 1.0);
        double tr = out;
        if (acc) {
            const float4 a = acc[row];
            tr = __dadd_ru(out, widen(a.x));
            if (flags) {
                const double lo_sum = row == fault_row ? 2.0 : widen(a.z);
                uint32_t f = 0;
                if (__dadd_rd(lo_sum, sl) > 1.0) f |= IMPACT_ROW_LO_SUM_ABOVE_ONE;
                if (__dadd_ru(__dadd_ru(widen(a.y), su), tr) < 1.0) f |= IMPACT_ROW_UP_SUM_BELOW_ONE;
                flags[row] = f;
                if (f) atomicOr(status, IMPACT_STATUS_UNSOUND);
            }
        }
        sink_lo[row] = sl;
        sink_up[row] = su;
        trunc[row] = tr;
    }
}

// setup_fp32 (builds whose images are nearly all distinct): one warp per 32/n
// rows of one build, one lane per (row, dimension). Each lane builds its
// dimension's table; the lanes of a row then exchange their maxima and sums
// by shuffles (finish_dim).
__global__ void __launch_bounds__(256, 3)
setup_fp32(const BatchIndex *__restrict__ B, uint32_t *__restrict__ status)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = warp0; u < B->units; u += nwarps) {
        const int q = find_problem(B->unit_begin, B->count, u);
        const ImpactDesc &D = *B->desc[q];
        if (D.share32) continue;
        const int n = D.n;
        const int rpw = 32 / n;
        const int slot = lane / n, d = lane - slot * n;
        const int64_t rows_q = B->row_begin[q + 1] - B->row_begin[q];
        const int64_t rl = (u - B->unit_begin[q]) * rpw + slot;
        const bool act = slot < rpw && rl < rows_q;
        unsigned char *rr = act ? B->rec[q] + rl * (int64_t)D.rec_stride : nullptr;
        DimOut o;
        if (act) {
            int idx[IMPACT_MAX_DIM], j;
            rowmath::decode_row(D, rl, idx, j);
            o = setup_dim(D, rl, idx, j, d, rec_table(rr, n) + D.dim[d].rec_off, status);
            reinterpret_cast<float4 *>(B->terms[q])[rl * n + d] = term_of(o);
        }
        finish_dim(D, o, d, slot * n, act, rr);
    }
}

// The same for few rows: four lanes per (row, dimension), a unit's 32/n rows in
// parts of 8/n.
__global__ void __launch_bounds__(128)
setup_split_fp32(const BatchIndex *__restrict__ B, uint32_t *__restrict__ status)
{
    constexpr int G = 4, kParts = 6;   // (32/n) / (8/n) rounded up, at most
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = warp0; v < B->units * kParts; v += nwarps) {
        const int64_t u = v / kParts;
        const int q = find_problem(B->unit_begin, B->count, u);
        const ImpactDesc &D = *B->desc[q];
        if (D.share32) continue;
        const int n = D.n;
        const int rpw = 32 / n, rpp = 32 / (G * n);
        const int slot = lane / (G * n), d = (lane - slot * G * n) / G;
        const int r = (int)(v - u * kParts) * rpp + slot;   // row of the unit
        if (r - slot >= rpw) continue;
        const int64_t rows_q = B->row_begin[q + 1] - B->row_begin[q];
        const int64_t rl = (u - B->unit_begin[q]) * rpw + r;
        const bool act = slot < rpp && r < rpw && rl < rows_q;
        unsigned char *rr = act ? B->rec[q] + rl * (int64_t)D.rec_stride : nullptr;
        int idx[IMPACT_MAX_DIM], j = 0;
        if (act) rowmath::decode_row(D, rl, idx, j);
        const DimOut o = setup_dim_split<G>(D, rl, idx, j, d,
                                            act ? rec_table(rr, n) + D.dim[d].rec_off : nullptr,
                                            status, act);
        const bool head = act && (lane & (G - 1)) == 0;
        if (head) reinterpret_cast<float4 *>(B->terms[q])[rl * n + d] = term_of(o);
        finish_dim(D, o, d, slot * G * n, head, rr, G);
    }
}

// items_fp32: the window and factor table of every distinct image
// (impact_desc.h), one lane or (few items, ImpactDim.group) eight lanes each:
// DimOut, then the window's (U, L) pairs.
__device__ __forceinline__ float2 *item_table(unsigned char *it)
{
    return reinterpret_cast<float2 *>(it + sizeof(DimOut));
}

__global__ void __launch_bounds__(128)
items_fp32(const BatchIndex *__restrict__ B, uint32_t *__restrict__ status)
{
    const int64_t total = B->item_units * 32;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {   // a warp's lanes share a unit
        const int seg = find_problem(B->item_begin, B->count * IMPACT_MAX_DIM, i >> 5);
        const int q = seg / IMPACT_MAX_DIM, d = seg % IMPACT_MAX_DIM;
        const ImpactDesc &D = *B->desc[q];
        const ImpactDim &g = D.dim[d];
        if (g.group == 8) {
            const int64_t c = (i - B->item_begin[seg] * 32) / 8;
            const bool act = c < g.n_items;
            int idx[IMPACT_MAX_DIM], j = 0;
            if (act) rowmath::decode_item(D, d, c, idx, j);
            unsigned char *it = B->items[q] + g.item_off + c * g.item_stride;
            const DimOut o = setup_dim_split<8>(D, c, idx, j, d, item_table(it), status, act);
            if (act && (i & 7) == 0) *reinterpret_cast<DimOut *>(it) = o;
            continue;
        }
        const int64_t c = i - B->item_begin[seg] * 32;
        if (c >= g.n_items) continue;
        int idx[IMPACT_MAX_DIM], j;
        rowmath::decode_item(D, d, c, idx, j);
        unsigned char *it = B->items[q] + g.item_off + c * g.item_stride;
        *reinterpret_cast<DimOut *>(it) = setup_dim(D, c, idx, j, d, item_table(it), status);
    }
}

// rows_fp32 (builds that share windows): the lanes of setup_fp32 load their
// dimension's item instead of making it, and the warp then copies the trimmed
// tables into the records, eight lanes per table in 16-byte pieces (items and
// record tables start 16-byte aligned). Bound by the records it writes.
__global__ void __launch_bounds__(256)
rows_fp32(const BatchIndex *__restrict__ B)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = warp0; u < B->units; u += nwarps) {
        const int q = find_problem(B->unit_begin, B->count, u);
        const ImpactDesc &D = *B->desc[q];
        if (!D.share32) continue;
        const int n = D.n;
        const int rpw = 32 / n;
        const int slot = lane / n, d = lane - slot * n;
        const int64_t rows_q = B->row_begin[q + 1] - B->row_begin[q];
        const int64_t rl = (u - B->unit_begin[q]) * rpw + slot;
        const bool act = slot < rpw && rl < rows_q;
        unsigned char *rr = act ? B->rec[q] + rl * (int64_t)D.rec_stride : nullptr;
        DimOut o;
        const float4 *src = nullptr;
        float4 *dst = nullptr;
        int pieces = 0;
        if (act) {
            int idx[IMPACT_MAX_DIM], j;
            rowmath::decode_row(D, rl, idx, j);
            const ImpactDim &g = D.dim[d];
            unsigned char *it = B->items[q] + g.item_off +
                                rowmath::item_of(D, rl, idx, j, d) * g.item_stride;
            o = *reinterpret_cast<const DimOut *>(it);
            const int p0 = o.f0 >> 1;
            pieces = ((o.f0 + o.tw + 1) >> 1) - p0;
            src = reinterpret_cast<const float4 *>(item_table(it)) + p0;
            dst = reinterpret_cast<float4 *>(rec_table(rr, n) + g.rec_off) + p0;
            if (d == 0) rec_row(rr, n)->leaf = leaf_of_row(D, idx, j);
        }
        finish_dim(D, o, d, slot * n, act, rr);
#pragma unroll
        for (int p0 = 0; p0 < 32; p0 += 4) {
            const int p = p0 + (lane >> 3);
            const float4 *s = reinterpret_cast<const float4 *>(
                __shfl_sync(0xffffffffu, (unsigned long long)src, p));
            float4 *t = reinterpret_cast<float4 *>(
                __shfl_sync(0xffffffffu, (unsigned long long)dst, p));
            const int k = __shfl_sync(0xffffffffu, pieces, p);
            for (int i = lane & 7; i < k; i += 8) t[i] = s[i];
        }
    }
}

// ---------------------------------------------------------------------------
// the walk
// ---------------------------------------------------------------------------

constexpr int kCap = IMPACT_WALK_CAP;      // nodes per level list (one chunk)
constexpr int kSlots = kCap + 1;           // and a spare slot
constexpr int kClaimBytes = 16;            // per warp: the claimed row range
constexpr int kTrimMin = 512;              // emit: candidates of a chunk worth trimming its table for

// Warp shared memory: a record buffer of the batch's largest record (in the count
// pass two: the row being walked and the next one, copied in meanwhile), then the work
// space (offsets fixed per problem by leaf_cap):
//   h      RecDim[n]                 the row record's per-dimension entries
//   ul     (U, L) x tsum_cap         the record's window tables
//   work   (n - 2) x kSlots x 12 B   node lists of levels 0..n-3
//   leaf   count: 8 x (leaf_cap + 1) words, the leaf table (see Leaf) with its
//          sorted form and sums; emit: twice 3 words per entry, the staged
//          table and its copy trimmed per chunk
struct WarpMem {
    RecDim *h;
    float2 *ul;
    unsigned char *work;
    float *leaf;
    int leaf_cap;
};

__host__ __device__ constexpr int align16(int x) { return (x + 15) & ~15; }

// Node lists of levels 0..n-3, padded to 16 bytes: the warp blocks are laid
// end to end and each starts with 16-byte record copies.
__host__ __device__ inline int list_bytes(int n) { return align16((n > 2 ? n - 2 : 0) * kSlots * 12); }

// Entries of an emit leaf table, even: the tables are 8-byte aligned.
__host__ __device__ constexpr int emit_cap(int leaf_cap) { return (leaf_cap + 1) & ~1; }

// Emit by lists (builds with shared leaf tables, rows of kListMin to kListMax
// entries): the leaf block of a row -- sorted upper factors, then U, L and column
// of the entries in C order, kListMax words each, and for every kept count k
// the k largest entries in C order, one byte each -- then the parents of a
// chunk and the chunk's start bits. Below 20 entries a parent's search costs
// more than the candidates that its list saves (building 6^7, 9 entries: 4.9 ms
// by lists, 4.3 by candidates), above 48 the lists outgrow the block. The window
// bound of a build (its rows' tables hold about a third of it) tells which side
// most rows are on: outside kListCapMin..kListCapMax entries the smaller blocks
// are worth more.
constexpr int kListMin = 20, kListMax = 48, kListCapMin = 64, kListCapMax = 160;
__host__ __device__ constexpr int list_block(int nb)   // bytes, multiple of 16
{
    return align16(16 * kListMax + nb * (nb + 1) / 2);
}
constexpr int kInfoBytes = 16 * kCap;
constexpr int kStartWords = kCap * kListMax / 32;

// Shared memory of the emit's leaf: the staged table and its trimmed copy, or a
// list block with the parents and start bits behind it.
__host__ __device__ inline int emit_leaf_bytes(int leaf_cap, bool lists)
{
    const int staged = align16(24 * emit_cap(leaf_cap));
    if (!lists) return staged;
    const int block = list_block(kListMax);
    return (staged > block ? staged : block) + kInfoBytes + 4 * kStartWords;
}

__device__ __forceinline__ WarpMem carve(unsigned char *work, unsigned char *rec, int n, int leaf_cap)
{
    WarpMem m;
    m.h = reinterpret_cast<RecDim *>(rec);
    m.ul = rec_table(rec, n);
    m.work = work;
    m.leaf = reinterpret_cast<float *>(m.work + list_bytes(n));
    m.leaf_cap = leaf_cap;
    return m;
}

// Level k node list: P (RU product of upper factors), Pl (RD product of lower
// factors), col (column of the prefix).
struct NodeList {
    float *P, *Pl;
    int *col;
};

__device__ __forceinline__ NodeList node_list(unsigned char *work, int k)
{
    NodeList L;
    // kCap nodes and one spare slot that takes the stores of the lanes
    // whose candidate was not kept (stores without a branch)
    unsigned char *b = work + k * (kSlots * 12);
    L.P = reinterpret_cast<float *>(b);
    L.Pl = L.P + kSlots;
    L.col = reinterpret_cast<int *>(L.Pl + kSlots);
    return L;
}

// Per-lane partial sums of the count walk (rounded outward, FP32): pairs
// kept, upper-bound mass of the dropped in-window targets, and the sums of
// the kept pairs' upper and lower bounds (row checks). All terms are
// non-negative, so the sums are bounds with a relative excess of at most a
// few units of 2^-23.
struct CountAcc {
    int cnt = 0;
    float drop = 0.0f, sup = 0.0f, slo = 0.0f;
};

// Where the emit walk writes: the row's len pairs, the arrays offset to its
// first pair.
struct EmitOut {
    int32_t *col;
    float *lo, *up;
    int len;
};

// The leaf table of a row: the last two dimensions m = n - 2 and l = n - 1
// (dimension 0 alone when n = 1) as one list of entries j = a * tw_l + b in C
// order: bu[j] = RU(U_m[a] U_l[b]), bl[j] = RD(L_m[a] L_l[b]) and the column
// offset bc[j] = cb_m + a stride_m + cb_l + b. For the count pass also the
// entries sorted by bu descending (su, with their bl in sl) and the sums
// pu[k] = RU sum of su[0..k), pl[k] = RD sum of sl[0..k), sf[k] = RU sum of
// su[k..nb). Staged when nb <= leaf_cap, else evaluated where needed.
struct Leaf {
    float tot_u, tot_l;   // count pass: RU sum of bu and RD sum of bl over all entries
    int nb;        // entries
    int tw_l;      // width of the last dimension (b runs fastest)
    uint32_t magic_l;
    bool staged;
    bool sorted;          // count pass: su, sl, pu, pl, sf are built
    const float4 *shared;    // count pass: the row's shared sorted table, or null
    uint32_t magic_nb;    // ceil(2^32 / nb) when 1 < nb <= 4096, for the emit's flat layout
    float *bu, *bl, *su, *sl, *pu, *pl, *sf;
    int *bc;
};

__device__ __forceinline__ Leaf leaf_of(const WarpMem &S, int n)
{
    Leaf f;
    const RecDim &hl = S.h[n - 1];
    f.tw_l = hl.tw;
    f.magic_l = hl.magic;
    f.nb = n >= 2 ? S.h[n - 2].tw * hl.tw : hl.tw;
    f.staged = f.nb <= S.leaf_cap;
    f.sorted = false;
    f.shared = nullptr;
    f.magic_nb = (f.nb > 1 && f.nb <= 4096)   // ceil(2^32 / nb)
                     ? 0xffffffffu / (unsigned)f.nb + 1u : 0u;
    const int c = S.leaf_cap + 1;
    f.bu = S.leaf;
    f.bl = f.bu + c;
    f.bc = reinterpret_cast<int *>(f.bl + c);
    f.su = reinterpret_cast<float *>(f.bc + c);
    f.sl = f.su + c;
    f.pu = f.sl + c;
    f.pl = f.pu + c;
    f.sf = f.pl + c;
    return f;
}

// Entry j of the leaf table, evaluated from the record's tables.
struct LeafEntry {
    float u, l;
    int c;
};

__device__ __forceinline__ LeafEntry leaf_eval(const WarpMem &S, int n, const Leaf &f, int j)
{
    const RecDim &hl = S.h[n - 1];
    LeafEntry e;
    if (n == 1) {
        const float2 v = S.ul[hl.tb + j];
        e.u = v.x;
        e.l = v.y;
        e.c = hl.cb + j;
        return e;
    }
    const RecDim &hm = S.h[n - 2];
    const int a = f.tw_l > 1 ? (int)__umulhi((uint32_t)j, f.magic_l) : j;
    const int b = j - a * f.tw_l;
    const float2 vm = S.ul[hm.tb + a], vl = S.ul[hl.tb + b];
    e.u = __fmul_ru(vm.x, vl.x);
    e.l = __fmul_rd(vm.y, vl.y);
    e.c = hm.cb + a * hm.stride + hl.cb + b;
    return e;
}

// Inclusive warp scans of a lane's value with directed rounding (a fixed
// association: the same bits whatever ran before).
__device__ __forceinline__ float scan_ru(float x, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = __fadd_ru(x, y);
    }
    return x;
}
__device__ __forceinline__ float scan_rd(float x, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = __fadd_rd(x, y);
    }
    return x;
}

// Count pass: stages the leaf table of a row with its sorted form and sums when
// it fits (dense rows: only the totals). A row of at most two dimensions has
// one parent (the root): testing its entries directly costs less than sorting
// them.
__device__ void leaf_build(const WarpMem &S, int n, Leaf &f, int lane, float cut)
{
    if (n <= 2 && cut > 0.0f) return;
    float su_l = 0.0f, sl_l = 0.0f;   // this lane's part of the totals
    for (int j = lane; j < f.nb; j += 32) {
        const LeafEntry e = leaf_eval(S, n, f, j);
        if (f.staged) {
            f.bu[j] = e.u;
            f.bl[j] = e.l;
            f.bc[j] = e.c;
        }
        su_l = __fadd_ru(su_l, e.u);
        sl_l = __fadd_rd(sl_l, e.l);
    }
    __syncwarp();
    if (!(cut > 0.0f)) {   // the totals serve the dense count only
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            su_l = __fadd_ru(su_l, __shfl_xor_sync(0xffffffffu, su_l, o));
            sl_l = __fadd_rd(sl_l, __shfl_xor_sync(0xffffffffu, sl_l, o));
        }
        f.tot_u = __shfl_sync(0xffffffffu, su_l, 0);
        f.tot_l = __shfl_sync(0xffffffffu, sl_l, 0);
    }
    if (!f.staged || !(cut > 0.0f)) return;
    f.sorted = true;
    if (f.nb <= 32) {
        // one entry per lane: a bitonic sorting network over the warp puts
        // the entry of rank r (bu descending, ties by index) in lane r, then
        // scans in registers give the sums. The sort key is the bits of bu
        // inverted (bu >= 0, so its bits grow with it) above the index:
        // ascending keys are bu descending, ties by index; lanes past the
        // table hold the largest key and sort last.
        const bool in = lane < f.nb;
        unsigned long long key = ~0ull;
        if (in)
            key = ((unsigned long long)(~__float_as_uint(f.bu[lane])) << 32) | (unsigned)lane;
#pragma unroll
        for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
            for (int jj = k >> 1; jj > 0; jj >>= 1) {
                const unsigned long long pk = __shfl_xor_sync(0xffffffffu, key, jj);
                const bool want_first = ((lane & jj) == 0) == ((lane & k) == 0);
                if (want_first != (key < pk)) key = pk;
            }
        }
        const float u = in ? __uint_as_float(~(unsigned)(key >> 32)) : 0.0f;
        const float lv = in ? f.bl[(int)(key & 0xffffffffu)] : 0.0f;
        const float ux = u;
        const float iu = scan_ru(ux, lane);
        const float il = scan_rd(lv, lane);
        float su_ = ux;   // suffix sums, rounded up
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float y = __shfl_down_sync(0xffffffffu, su_, o);
            if (lane + o < 32) su_ = __fadd_ru(su_, y);
        }
        if (lane < f.nb) {
            f.su[lane] = u;
            f.pu[lane + 1] = iu;
            f.pl[lane + 1] = il;
            f.sf[lane] = su_;
        }
        if (lane == 0) {
            f.pu[0] = 0.0f;
            f.pl[0] = 0.0f;
            f.sf[f.nb] = 0.0f;
        }
        __syncwarp();
        return;
    }
    // rank of entry j by bu descending (ties by index): its sorted position
    for (int j = lane; j < f.nb; j += 32) {
        const float u = f.bu[j];
        int r = 0;
        for (int i = 0; i < f.nb; ++i) {
            const float v = f.bu[i];
            r += (v > u) || (v == u && i < j);
        }
        f.su[r] = u;
        f.sl[r] = f.bl[j];
    }
    __syncwarp();
    // prefix sums in sorted order (pu, pl: entries 0..k-1 -> index k) and
    // suffix sums (sf[k]: entries k..nb-1), rounded outward
    float cu = 0.0f, cl = 0.0f;
    for (int k0 = 0; k0 < f.nb; k0 += 32) {
        const int k = k0 + lane;
        const float u = k < f.nb ? f.su[k] : 0.0f;
        const float l = k < f.nb ? f.sl[k] : 0.0f;
        const float iu = __fadd_ru(scan_ru(u, lane), cu);
        const float il = __fadd_rd(scan_rd(l, lane), cl);
        if (k < f.nb) {
            f.pu[k + 1] = iu;
            f.pl[k + 1] = il;
        }
        cu = __shfl_sync(0xffffffffu, iu, 31);
        cl = __shfl_sync(0xffffffffu, il, 31);
    }
    if (lane == 0) {
        f.pu[0] = 0.0f;
        f.pl[0] = 0.0f;
    }
    float cs = 0.0f;   // suffix sums, from the end
    for (int k1 = f.nb; k1 > 0; k1 -= 32) {
        const int k = k1 - 1 - lane;
        const float u = k >= 0 ? f.su[k] : 0.0f;
        const float iu = __fadd_ru(scan_ru(u, lane), cs);
        if (k >= 0) f.sf[k] = iu;
        cs = __shfl_sync(0xffffffffu, iu, 31);
    }
    if (lane == 0) f.sf[f.nb] = 0.0f;
    __syncwarp();
}

// leaf_fp32: the sorted leaf table of every distinct image of the last two
// dimensions together, one warp each, from their items: {nb, ..} in 16 bytes,
// then (su, sf, pu, pl) per entry k = 0..nb, su[nb] unused, and the list block of
// the emit pass. Tables of more than leaf_cap entries stay empty (their rows
// test the entries directly).
struct LeafHead {
    int nb, pad[3];
};

// Where the list block of a leaf table stands.
__host__ __device__ constexpr int leaf_lists_at(int leaf_cap)
{
    return (int)sizeof(LeafHead) + 16 * (leaf_cap + 1);
}

__global__ void __launch_bounds__(128)
leaf_fp32(const BatchIndex *__restrict__ B, int warp_smem)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    unsigned char *const mine = smem_raw + (size_t)(threadIdx.x >> 5) * warp_smem;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = warp0; u < B->leaf_total; u += nwarps) {
        const int q = find_problem(B->leaf_begin, B->count, u);
        const ImpactDesc &D = *B->desc[q];
        const int n = D.n;
        const int64_t c0 = u - B->leaf_begin[q];
        int idx[IMPACT_MAX_DIM], j;
        {
            int64_t c = c0;
            j = D.leaf_rep[(int)(c % D.leaf_classes)];
            c /= D.leaf_classes;
#pragma unroll
            for (int k = IMPACT_MAX_DIM - 1; k >= 0; --k) {
                idx[k] = 0;
                if (k < n && D.leaf_mul[k] != 0) {
                    idx[k] = (int)(c % D.dim[k].N);
                    c /= D.dim[k].N;
                }
            }
        }
        // the entries of the last two dimensions of a record, in place
        WarpMem S;
        S.h = reinterpret_cast<RecDim *>(mine) - (n - 2);
        S.ul = reinterpret_cast<float2 *>(mine + 2 * sizeof(RecDim));
        const int wm = (D.dim[n - 2].wcap + 1) & ~1, wl = (D.dim[n - 1].wcap + 1) & ~1;
        S.work = nullptr;
        S.leaf = reinterpret_cast<float *>(S.ul + wm + wl);
        S.leaf_cap = D.leaf_cap;
        for (int e = 0; e < 2; ++e) {
            const int d = n - 2 + e;
            const ImpactDim &g = D.dim[d];
            unsigned char *it = B->items[q] + g.item_off +
                                rowmath::item_of(D, 0, idx, j, d) * g.item_stride;
            const DimOut o = *reinterpret_cast<const DimOut *>(it);
            if (lane == 0) {
                RecDim rd;
                rd.tw = o.tw;
                rd.tb = e * wm;
                rd.cb = (o.a + o.f0) * g.stride;
                rd.magic = o.tw > 1
                               ? (uint32_t)((0x100000000ull + (unsigned)o.tw - 1) / (unsigned)o.tw) : 0u;
                rd.cp = rd.SR = 0.0f;
                rd.stride = g.stride;
                rd.lay = 0;
                S.h[d] = rd;
            }
            for (int k = lane; k < o.tw; k += 32) S.ul[e * wm + k] = item_table(it)[o.f0 + k];
        }
        __syncwarp();
        unsigned char *out = B->leaf[q] + c0 * D.leaf_stride;
        Leaf f = leaf_of(S, n);
        if (f.nb > 0 && f.staged) leaf_build(S, n, f, lane, D.cutoff32);
        if (lane == 0) reinterpret_cast<LeafHead *>(out)->nb = f.sorted ? f.nb : -1;
        if (f.sorted) {
            float4 *to = reinterpret_cast<float4 *>(out + sizeof(LeafHead));
            for (int k = lane; k <= f.nb; k += 32)
                to[k] = make_float4(k < f.nb ? f.su[k] : 0.0f, f.sf[k], f.pu[k], f.pl[k]);
        }
        if (D.lists && f.sorted && f.nb >= kListMin && f.nb <= kListMax) {   // the emit's list block
            const int nb = f.nb;
            float *const block = reinterpret_cast<float *>(mine + warp_smem - list_block(kListMax));
            unsigned char *const lists = reinterpret_cast<unsigned char *>(block + 4 * kListMax);
            // sorted positions of entries lane and lane + 32 (ties by index)
            const bool h0 = lane < nb, h1 = lane + 32 < nb;
            const float u0 = h0 ? f.bu[lane] : 0.0f, u1 = h1 ? f.bu[lane + 32] : 0.0f;
            int r0 = 0, r1 = 0;
            for (int i = 0; i < nb; ++i) {
                const float v = f.bu[i];
                r0 += v > u0 || (v == u0 && i < lane);
                r1 += v > u1 || (v == u1 && i < lane + 32);
            }
            if (!h0) r0 = INT_MAX;
            if (!h1) r1 = INT_MAX;
            for (int j = lane; j < kListMax; j += 32) {
                const bool in = j < nb;
                block[j] = in ? f.su[j] : 0.0f;
                block[j + kListMax] = in ? f.bu[j] : 0.0f;
                block[j + 2 * kListMax] = in ? f.bl[j] : 0.0f;
                block[j + 3 * kListMax] = in ? __int_as_float(f.bc[j]) : 0.0f;
            }
            for (int k = 1; k <= nb; ++k) {
                unsigned char *const l = lists + k * (k - 1) / 2;
                const unsigned b0 = __ballot_sync(0xffffffffu, r0 < k);
                if (r0 < k) l[__popc(b0 & lanemask_lt())] = (unsigned char)lane;
                if (nb > 32) {
                    const unsigned b1 = __ballot_sync(0xffffffffu, r1 < k);
                    if (r1 < k) l[__popc(b0) + __popc(b1 & lanemask_lt())] = (unsigned char)(lane + 32);
                }
            }
            __syncwarp();
            float4 *const to = reinterpret_cast<float4 *>(out + leaf_lists_at(D.leaf_cap));
            for (int i = lane; i < (list_block(nb) >> 4); i += 32)
                to[i] = reinterpret_cast<const float4 *>(block)[i];
        }
        __syncwarp();
    }
}

// Node of a level list, or the root (P = Pl = 1, column 0).
struct Node {
    float P, Pl;
    int c;
};

__device__ __forceinline__ Node node_at(const NodeList &L, bool root, int i)
{
    if (root) return Node{1.0f, 1.0f, 0};
    return Node{L.P[i], L.Pl[i], L.col[i]};
}

// A narrow window (tw <= 32) is walked with each lane fixed on one target t
// of it: the warp holds floor(32 / tw) parents at a time, lane = slot * tw + t
// (slot-major, so ballot order is C order), and the lane's factors and
// column offset stay in registers. Wider windows are walked flat: candidate e
// = parent * tw + t, one lane each.
struct Lanes {
    int slots;     // parents per warp step (narrow), 0: flat
    int slot, t;   // this lane's slot and target (narrow)
    bool on;       // this lane holds a candidate slot (narrow)
};

__device__ __forceinline__ Lanes lanes_of(const RecDim &h, int lane)
{
    Lanes z{0, 0, 0, false};
    if (h.lay != 0) {
        z.slots = h.lay & 0xffff;
        z.slot = h.tw > 1 ? (int)__umulhi((uint32_t)lane, h.magic) : lane;
        z.t = lane - z.slot * h.tw;
        z.on = z.slot < z.slots;
    }
    return z;
}

// Candidates per chunk of a level list: whole parents when the window is
// narrow (the narrow walk steps over parents), else kCap.
__device__ __forceinline__ int chunk_of(const RecDim &h)
{
    return h.lay != 0 ? (h.lay >> 16) : kCap;
}

// Children of candidates [c0, c1) of the level k - 1 list (the root when
// k = 0) in dimension k, kept ones compacted into the level k list in order.
// A candidate e is (parent e / tw, target t = e mod tw of the trimmed window).
template <bool COUNT>
__device__ __forceinline__ int expand(const WarpMem &S, int k, bool root, int c0, int c1, int lane,
                                      CountAcc &acc)
{
    const RecDim &h = S.h[k];
    const int tw = h.tw, tb = h.tb, cb = h.cb, st = h.stride;
    const uint32_t magic = h.magic;
    const float cp = h.cp, SR = COUNT ? h.SR : 0.0f;
    const NodeList Lc = node_list(S.work, k);
    const NodeList Lp = node_list(S.work, root ? 0 : k - 1);
    const Lanes z = lanes_of(h, lane);
    int nout = 0;
    __syncwarp();   // the list's readers are done
    auto offer = [&](bool act, const Node &par, float2 ul, int t) {
        const float Pc = __fmul_ru(par.P, ul.x);
        const bool keep = act && Pc >= cp;
        if (COUNT) {
            const float d = __fadd_ru(acc.drop, __fmul_ru(Pc, SR));
            acc.drop = (act && !keep) ? d : acc.drop;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        const int o = keep ? nout + __popc(bal & lanemask_lt()) : kCap;
        Lc.P[o] = Pc;
        Lc.Pl[o] = __fmul_rd(par.Pl, ul.y);
        Lc.col[o] = par.c + cb + t * st;
        nout += __popc(bal);
    };
    if (z.slots > 0) {   // narrow: c0, c1 are multiples of tw
        const int p0 = tw > 1 ? (int)__umulhi((uint32_t)c0, magic) : c0;
        const int p1 = tw > 1 ? (int)__umulhi((uint32_t)c1, magic) : c1;
        const float2 ul = z.on ? S.ul[tb + z.t] : make_float2(0.0f, 0.0f);
        for (int pb = p0; pb < p1; pb += z.slots) {
            const int pi = pb + z.slot;
            const bool act = z.on && pi < p1;
            offer(act, act ? node_at(Lp, root, pi) : Node{0.0f, 0.0f, 0}, ul, z.t);
        }
    } else {
        for (int e0 = c0; e0 < c1; e0 += 32) {
            const int e = e0 + lane;
            const bool act = e < c1;
            const int pi = (int)__umulhi((uint32_t)e, magic);
            const int t = e - pi * tw;
            offer(act, act ? node_at(Lp, root, pi) : Node{0.0f, 0.0f, 0},
                  act ? S.ul[tb + t] : make_float2(0.0f, 0.0f), t);
        }
    }
    __syncwarp();
    return nout;
}


// Bounds of the sum of k emitted products RU(P x_i) (up) or RD(Pl y_i) (lo)
// from the RU / RD sum s of the x_i / y_i: each rounded product is within a
// relative 2^-23 (plus 2^-149 below the normal range) of the exact one.
__device__ __forceinline__ float up_sum(float P, float s, int k)
{
    return __fmaf_ru((float)k, 1.17549435e-38f, __fmul_ru(__fmul_ru(P, s), 1.00000095f));
}
__device__ __forceinline__ float lo_sum(float Pl, float s, int k)
{
    return fmaxf(__fmaf_rd(-(float)k, 1.17549435e-38f, __fmul_rd(__fmul_rd(Pl, s), 0.99999905f)),
                 0.0f);
}

// Count pass over the leaves of npar parents (a level n - 3 list, or the
// root): pairs, their up and lo sums and the upper bound of the dropped
// mass, per lane (one lane per parent).
__device__ void leaf_count(const WarpMem &S, int n, const Leaf &f, const NodeList &Lp, bool root,
                           int npar, int lane, CountAcc &acc, float cut)
{
    const int nb = f.nb;
    if (!(cut > 0.0f)) {   // dense: every entry is kept
        for (int pi = lane; pi < npar; pi += 32) {
            const Node par = node_at(Lp, root, pi);
            acc.cnt += nb;
            acc.sup = __fadd_ru(acc.sup, up_sum(par.P, f.tot_u, nb));
            acc.slo = __fadd_rd(acc.slo, lo_sum(par.Pl, f.tot_l, nb));
        }
        return;
    }
    if (f.sorted) {
        // the kept entries of a parent are a prefix of the sorted table:
        // RU(P su[k]) >= cut for k below the count, not above it
        for (int pi = lane; pi < npar; pi += 32) {
            const Node par = node_at(Lp, root, pi);
            int lo = 0, hi = nb;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (__fmul_ru(par.P, f.su[mid]) >= cut) lo = mid + 1;
                else hi = mid;
            }
            acc.cnt += lo;
            acc.sup = __fadd_ru(acc.sup, up_sum(par.P, f.pu[lo], lo));
            acc.slo = __fadd_rd(acc.slo, lo_sum(par.Pl, f.pl[lo], lo));
            acc.drop = __fadd_ru(acc.drop, __fmul_ru(par.P, f.sf[lo]));
        }
        return;
    }
    // the root's table, or a table too wide to stage: every entry under
    // every parent
    for (int pi = 0; pi < npar; ++pi) {
        const Node par = node_at(Lp, root, pi);
        for (int j0 = 0; j0 < nb; j0 += 32) {
            const int j = j0 + lane;
            if (j < nb) {
                const LeafEntry e = leaf_eval(S, n, f, j);
                const float Pc = __fmul_ru(par.P, e.u);
                if (Pc >= cut) {
                    acc.cnt += 1;
                    acc.sup = __fadd_ru(acc.sup, Pc);
                    acc.slo = __fadd_rd(acc.slo, __fmul_rd(par.Pl, e.l));
                } else {
                    acc.drop = __fadd_ru(acc.drop, Pc);
                }
            }
        }
    }
}

// The same from the row's shared leaf table (in L2; the searches of a step's
// parents overlap).
__device__ __forceinline__ void leaf_count_shared(const float4 *__restrict__ tab, int nb,
                                                  const NodeList &Lp, int npar, int lane,
                                                  CountAcc &acc, float cut)
{
    for (int pi = lane; pi < npar; pi += 32) {
        const float P = Lp.P[pi], Pl = Lp.Pl[pi];
        int lo = 0, hi = nb;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (__fmul_ru(P, __ldg(&tab[mid].x)) >= cut) lo = mid + 1;
            else hi = mid;
        }
        const float4 e = __ldg(tab + lo);
        acc.cnt += lo;
        acc.sup = __fadd_ru(acc.sup, up_sum(P, e.z, lo));
        acc.slo = __fadd_rd(acc.slo, lo_sum(Pl, e.w, lo));
        acc.drop = __fadd_ru(acc.drop, __fmul_ru(P, e.y));
    }
}

// Stores of one pair that the predicate guards, without a branch around them.
__device__ __forceinline__ void st_pair(bool p, int32_t *c, float *l, float *u, int32_t col, float lo,
                                        float up)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %0, 0;\n\t"
                 "@q st.global.b32 [%1], %4;\n\t@q st.global.b32 [%2], %5;\n\t"
                 "@q st.global.b32 [%3], %6;\n\t}"
                 :: "r"((int)p), "l"(c), "l"(l), "l"(u), "r"(col), "r"(__float_as_int(lo)),
                    "r"(__float_as_int(up)) : "memory");
}

// One candidate per lane: the kept ones are compacted in lane order after the
// pairs already written and stored (predicated, no divergence).
__device__ __forceinline__ void offer_pair(bool act, float P, float Pl, int c, float u, float l,
                                           float cut, const EmitOut &out, int &written)
{
    const float Pc = __fmul_ru(P, u);
    const bool keep = act && Pc >= cut;
    const unsigned bal = __ballot_sync(0xffffffffu, keep);
    const int pos = written + __popc(bal & lanemask_lt());
    st_pair(keep && pos < out.len, out.col + pos, out.lo + pos, out.up + pos, c, __fmul_rd(Pl, l), Pc);
    written += __popc(bal);
}

// The leaf table as the emit pass walks it: the products of upper and of lower
// factors and the columns, `cap` words apart (32-bit arrays: the lanes of a step
// wrap from a parent's last entry to the next one's first, which pairs of
// words in one array turn into bank conflicts).
struct EmitLeaf {
    float *u;
    int cap;
    int nb;
    uint32_t magic;    // ceil(2^32 / nb)
    bool staged;
};

__device__ __forceinline__ EmitLeaf emit_leaf(const WarpMem &S, const Leaf &f)
{
    EmitLeaf e;
    e.u = S.leaf;
    e.cap = emit_cap(S.leaf_cap);
    e.nb = f.nb;
    e.magic = f.magic_nb;
    e.staged = f.staged;
    return e;
}

// Emit pass over the leaves of npar parents from the staged table: each entry
// under each parent one lane (flat: candidate e = parent * nb + entry, so no
// lane idles but in the last step); kept pairs are compacted in C order and
// stored warp-contiguously. A layout that keeps the table in registers and
// steps over parents measured slower: its lanes idle when 32 is not a multiple
// of nb, and its registers cost occupancy.
__device__ __forceinline__ void leaf_emit(const WarpMem &S, const EmitLeaf &f, const NodeList &Lp,
                                          int npar, int lane, const EmitOut &out, int &written,
                                          float cut)
{
    const float *tu = f.u;
    const int cs = f.cap;
    int nb = f.nb;
    uint32_t magic = f.magic;
    if (cut > 0.0f && npar * nb >= kTrimMin) {
        // entries that no parent of these can keep: RU(P x) is monotone in P,
        // so an entry below the cutoff under the largest P is below it under
        // every P. The rest, in C order, form the table walked below; the
        // pairs are the same. (A pass over the table and a division: worth it
        // only when the parents and the table are large.)
        float pm = 0.0f;
        for (int pi = lane; pi < npar; pi += 32) pm = fmaxf(pm, Lp.P[pi]);
        pm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(pm)));   // pm >= 0
        float *const su = f.u + 3 * cs;
        int nt = 0;
        for (int j0 = 0; j0 < nb; j0 += 32) {
            const int j = min(j0 + lane, nb - 1);
            const float v = tu[j];
            const bool k = j0 + lane < nb && __fmul_ru(pm, v) >= cut;
            const unsigned bal = __ballot_sync(0xffffffffu, k);
            if (k) {
                const int o = nt + __popc(bal & lanemask_lt());
                su[o] = v;
                su[o + cs] = tu[j + cs];
                su[o + 2 * cs] = tu[j + 2 * cs];   // the column's bits
            }
            nt += __popc(bal);
        }
        __syncwarp();
        if (nt == 0) return;
        if (nt < nb) {
            nb = nt;
            magic = nt > 1 ? 0xffffffffu / (unsigned)nt + 1u : 0u;   // ceil(2^32 / nt)
            tu = su;
        }
    }
    // the division is exact for e < 64 nb, nb <= 4096; lanes past the end read
    // the last candidate and store nothing
    const int total = npar * nb;
    auto offer = [&](bool act, const Node &par, int j) {
        offer_pair(act, par.P, par.Pl, par.c + __float_as_int(tu[j + 2 * cs]), tu[j], tu[j + cs],
                   cut, out, written);
    };
    int e0 = 0;
    for (; e0 + 32 < total; e0 += 64) {   // two candidates per lane and step
        const int ea = e0 + lane, eb = min(e0 + 32 + lane, total - 1);
        const int pa = nb == 1 ? ea : (int)__umulhi((uint32_t)ea, magic);
        const int pb = nb == 1 ? eb : (int)__umulhi((uint32_t)eb, magic);
        const int ja = ea - pa * nb, jb = eb - pb * nb;
        const Node na = node_at(Lp, false, pa), nc = node_at(Lp, false, pb);
        const float ua = tu[ja], la = tu[ja + cs], ub = tu[jb], lb = tu[jb + cs];
        const int ca = __float_as_int(tu[ja + 2 * cs]), cb = __float_as_int(tu[jb + 2 * cs]);
        offer_pair(true, na.P, na.Pl, na.c + ca, ua, la, cut, out, written);
        offer_pair(e0 + 32 + lane < total, nc.P, nc.Pl, nc.c + cb, ub, lb, cut, out, written);
    }
    for (; e0 < total; e0 += 32) {
        const int e = min(e0 + lane, total - 1);
        const int pi = nb == 1 ? e : (int)__umulhi((uint32_t)e, magic);
        offer(e0 + lane < total, node_at(Lp, false, pi), e - pi * nb);
    }
}

// The same from the row's list block: a parent keeps the k largest entries of
// the table (RU(P x) is monotone in x), k from a search in the sorted table, and
// list k holds them in C order, so every lane of every step writes a pair: the
// chunk's pairs are numbered through, a bit marks each parent's first pair, and
// a pair's parent is the number of bits up to it. Steps of 32 pairs and not of
// 32 candidates (the 11^5 room: 62 and not 97 a row, about 27 instructions each
// and not 33), for about 80 instructions per 32 parents: its emit pass 7.45 ->
// 6.69 ms, the list blocks 0.2 ms of leaf_fp32.
__device__ __forceinline__ void emit_lists(unsigned char *block, unsigned char *after, int nb,
                                           const NodeList &Lp, int npar, int lane,
                                           const EmitOut &out, int &written, float cut)
{
    const float *const su = reinterpret_cast<const float *>(block);
    const unsigned char *const lists = block + 16 * kListMax;
    float4 *const info = reinterpret_cast<float4 *>(after);
    unsigned *const bits = reinterpret_cast<unsigned *>(after + kInfoBytes);
    int start[kCap / 32], total = 0, nord = 0;
    __syncwarp();   // the chunk before is written
#pragma unroll
    for (int h = 0; h < kCap / 32; ++h) {
        const int pi = lane + 32 * h;
        const float P = pi < npar ? Lp.P[pi] : 0.0f;
        int lo = 0, hi = nb;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (__fmul_ru(P, su[mid]) >= cut) lo = mid + 1; else hi = mid;
        }
        int s = lo;   // pairs up to this parent
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        const unsigned some = __ballot_sync(0xffffffffu, lo > 0);
        start[h] = lo > 0 ? total + s - lo : -1;
        if (lo > 0)
            info[nord + __popc(some & lanemask_lt())] =
                make_float4(P, Lp.Pl[pi], __int_as_float(Lp.col[pi]),
                            __int_as_float(lo * (lo - 1) / 2 - start[h]));
        total += __shfl_sync(0xffffffffu, s, 31);
        nord += __popc(some);
    }
    for (int w = lane; w < (total + 31) >> 5; w += 32) bits[w] = 0;
    __syncwarp();
#pragma unroll
    for (int h = 0; h < kCap / 32; ++h)
        if (start[h] >= 0) atomicOr(&bits[start[h] >> 5], 1u << (start[h] & 31));
    __syncwarp();
    const int room = min(total, out.len - written);
    int before = -1;   // parents whose first pair stands before this step, less one
    int32_t *const col = out.col + written;
    float *const lo = out.lo + written, *const up = out.up + written;
    const unsigned le = lanemask_lt() | (1u << lane);
    // two steps at once: a step is a chain of four shared-memory loads
    for (int o0 = 0; o0 < total; o0 += 64) {
        const unsigned wa = bits[o0 >> 5], wb = o0 + 32 < total ? bits[(o0 >> 5) + 1] : 0u;
        const int oa = o0 + lane, ob = oa + 32;
        const float4 pa = info[before + __popc(wa & le)];
        before += __popc(wa);
        const float4 pb = info[before + __popc(wb & le)];
        before += __popc(wb);
        const float *const ea = su + lists[__float_as_int(pa.w) + min(oa, total - 1)];
        const float *const eb = su + lists[__float_as_int(pb.w) + min(ob, total - 1)];
        const float ua = __fmul_ru(pa.x, ea[kListMax]), la = __fmul_rd(pa.y, ea[2 * kListMax]);
        const int ca = __float_as_int(pa.z) + __float_as_int(ea[3 * kListMax]);
        const float ub = __fmul_ru(pb.x, eb[kListMax]), lb = __fmul_rd(pb.y, eb[2 * kListMax]);
        const int cb = __float_as_int(pb.z) + __float_as_int(eb[3 * kListMax]);
        st_pair(oa < room, col + oa, lo + oa, up + oa, ca, la, ua);
        st_pair(ob < room, col + ob, lo + ob, up + ob, cb, lb, ub);
    }
    written += total;
}

// The same for a table too wide to stage, and for the root (rows of at most two
// dimensions): entries evaluated where they are read.
__device__ __forceinline__ void leaf_emit_wide(const WarpMem &S, int n, const Leaf &f,
                                               const NodeList &Lp, bool root, int npar, int lane,
                                               const EmitOut &out, int &written, float cut)
{
    for (int pi = 0; pi < npar; ++pi) {
        const Node par = node_at(Lp, root, pi);
        for (int j0 = 0; j0 < f.nb; j0 += 32) {
            const LeafEntry e = leaf_eval(S, n, f, min(j0 + lane, f.nb - 1));
            offer_pair(j0 + lane < f.nb, par.P, par.Pl, par.c + e.c, e.u, e.l, cut, out, written);
        }
    }
}

// Count walk: levels 0..n-3 of one row as node lists, depth first over chunks,
// the leaves under every chunk of the deepest list. LEFT lists are still to
// come; the recursion is unrolled at compile time (a loop with the level as a
// variable spends more on finding its place than on the nodes: the 8^5 room's
// count pass took 1251 instructions a row, and takes 861). Every chunk takes at
// least one of a list's candidates, so every loop ends (counting the steps
// cost the 7-D building's count 2.80 -> 3.04 ms).
template <int LEFT, bool ROOT>
__device__ __forceinline__ void count_levels(const WarpMem &S, int n, const Leaf &f, int npar,
                                             int lane, CountAcc &acc, float cut)
{
    const int k = n - 2 - LEFT;
    const int total = npar * S.h[k].tw, chunk = max(chunk_of(S.h[k]), 1);
#pragma unroll 1
    for (int c0 = 0; c0 < total; c0 += chunk) {
        const int nout = expand<true>(S, k, ROOT, c0, min(c0 + chunk, total), lane, acc);
        if constexpr (LEFT > 1) {
            count_levels<LEFT - 1, false>(S, n, f, nout, lane, acc, cut);
        } else {
            const NodeList L = node_list(S.work, k);
            if (f.shared) leaf_count_shared(f.shared, f.nb, L, nout, lane, acc, cut);
            else leaf_count(S, n, f, L, false, nout, lane, acc, cut);
        }
    }
}

// Counts one row whose record is in S (its leaf table built or shared).
__device__ __forceinline__ void count_row(const WarpMem &S, int n, const Leaf &f, int lane,
                                          CountAcc &acc, float cut)
{
    switch (n) {
    case 1:
    case 2: leaf_count(S, n, f, NodeList{}, true, 1, lane, acc, cut); break;
    case 3: count_levels<1, true>(S, n, f, 1, lane, acc, cut); break;
    case 4: count_levels<2, true>(S, n, f, 1, lane, acc, cut); break;
    case 5: count_levels<3, true>(S, n, f, 1, lane, acc, cut); break;
    case 6: count_levels<4, true>(S, n, f, 1, lane, acc, cut); break;
    case 7: count_levels<5, true>(S, n, f, 1, lane, acc, cut); break;
    default: count_levels<6, true>(S, n, f, 1, lane, acc, cut); break;
    }
}

// Writes the pairs of one row whose record is in S, or (COUNT: the one-pass walk,
// which does both) counts them: the same lists, with the level as a variable (the unrolled recursion keeps every level's loop state
// live, and the emit's inner loop needs the registers: 64 let 8 warps per
// scheduler hide its shared-memory latency; unrolled, the 11^5 room's emit
// pass took 7.8 ms against 7.45). Every turn of the loop fills a list from one
// candidate or more, runs the leaves of one or leaves one whose candidates are
// used up, so the loop ends (counting the steps cost the room's emit 0.2 of 6.6
// ms).
template <bool COUNT>
__device__ __forceinline__ void walk_row(const WarpMem &S, int n, const Leaf &f, bool lists,
                                         int after, int lane, CountAcc &acc, const EmitOut &out,
                                         int &written, float cut)
{
    if (n <= 2) {
        if (COUNT) leaf_count(S, n, f, NodeList{}, true, 1, lane, acc, cut);
        else leaf_emit_wide(S, n, f, NodeList{}, true, 1, lane, out, written, cut);
        return;
    }
    const EmitLeaf g = emit_leaf(S, f);
    if (!COUNT && g.staged && !lists)
        for (int j = lane; j < f.nb; j += 32) {
            const LeafEntry e = leaf_eval(S, n, f, j);
            g.u[j] = e.u;
            g.u[j + g.cap] = e.l;
            g.u[j + 2 * g.cap] = __int_as_float(e.c);
        }
    const int last = n - 3;      // deepest list level
    int my_cur = 0, my_sz = 0;   // lane k: next candidate of level k, size of list k
    int k = 0;
    while (true) {
        if (k == last + 1) {
            const NodeList L = node_list(S.work, last);
            const int npar = __shfl_sync(0xffffffffu, my_sz, last);
            unsigned char *const block = reinterpret_cast<unsigned char *>(S.leaf);
            if (COUNT) leaf_count(S, n, f, L, false, npar, lane, acc, cut);
            else if (lists) emit_lists(block, block + after, f.nb, L, npar, lane, out, written, cut);
            else if (g.staged) leaf_emit(S, g, L, npar, lane, out, written, cut);
            else leaf_emit_wide(S, n, f, L, false, npar, lane, out, written, cut);
            k = last;
            continue;
        }
        const int npar = k == 0 ? 1 : __shfl_sync(0xffffffffu, my_sz, k - 1);
        const int cur = __shfl_sync(0xffffffffu, my_cur, k);
        const int total = npar * S.h[k].tw;
        if (cur >= total) {
            if (k == 0) break;
            --k;
            continue;
        }
        const int end = min(cur + max(chunk_of(S.h[k]), 1), total);
        const int nout = expand<COUNT>(S, k, k == 0, cur, end, lane, acc);
        if (lane == k) {
            my_cur = end;
            my_sz = nout;
        }
        if (lane == k + 1) my_cur = 0;
        ++k;
    }
}

// ---------------------------------------------------------------------------
// row offsets by decoupled look-back, and the FP64 row terms
// ---------------------------------------------------------------------------

// Per-row look-back word: flag (bits 62-63: 0 not yet counted, 1 count
// only, 2 inclusive prefix) and value (bits 0-61).
constexpr unsigned long long kLbAgg = 1ull << 62;
constexpr unsigned long long kLbIncl = 2ull << 62;
constexpr unsigned long long kLbVal = (1ull << 62) - 1;

// Publishes the row's pair count and returns the number of pairs in the
// rows before it. A row waits only for rows that warps took before it from
// the ascending row counter; those are running and publish their counts
// without waiting on anything, so every wait ends. The wait is still bounded
// (spin_limit sleeps): on expiry, or once another warp has given up (`abort`),
// it sets the timeout status and returns false, and the row publishes no
// prefix (the rows after it give up in turn).
__device__ bool lookback(unsigned long long *lb, int64_t row, int64_t cnt, int lane,
                         unsigned *abort_flag, uint32_t *status, int spin_limit, bool stall,
                         int64_t &prefix)
{
    volatile unsigned long long *v = lb;
    volatile unsigned *ab = abort_flag;
    prefix = 0;
    if (lane == 0 && !stall) v[row] = (row == 0 ? +kLbIncl : +kLbAgg) | (unsigned long long)cnt;
    if (row == 0) return true;
    int64_t j = row - 1;   // window of rows j - 31 .. j, lane i at j - i
    int spins = 0;
    while (true) {
        const int64_t r = j - lane;
        unsigned long long w = +kLbIncl;   // before row 0: prefix 0
        if (r >= 0) w = v[r];
        const unsigned flag = (unsigned)(w >> 62);
        const unsigned incl = __ballot_sync(0xffffffffu, flag == 2u);
        const unsigned none = __ballot_sync(0xffffffffu, flag == 0u);
        // lanes up to the nearest inclusive prefix (all 32 if there is none)
        const unsigned upto = incl ? ((incl & (0u - incl)) << 1) - 1u : 0xffffffffu;
        if (none & upto) {
            int give_up = 0;
            if (lane == 0) give_up = (++spins > spin_limit) || (*ab != 0u);
            give_up = __shfl_sync(0xffffffffu, give_up, 0);
            if (give_up) {
                if (lane == 0) {
                    atomicOr(status, IMPACT_STATUS_TIMEOUT);
                    atomicExch(abort_flag, 1u);
                }
                return false;
            }
            __nanosleep(100);
            continue;
        }
        long long s = ((upto >> lane) & 1u) ? (long long)(w & kLbVal) : 0ll;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        prefix += s;
        if (incl) break;
        j -= 32;
    }
    if (lane == 0 && !stall) v[row] = kLbIncl | (unsigned long long)(prefix + cnt);
    return true;
}


__device__ __forceinline__ float warp_sum_ru(float x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = __fadd_ru(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
__device__ __forceinline__ float warp_sum_rd(float x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = __fadd_rd(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

// ---------------------------------------------------------------------------
// the walk kernel
// ---------------------------------------------------------------------------

// 16-byte asynchronous copy global -> shared (both 16-byte aligned), and its
// group fences.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prior() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The problem of global row x, searched from problem q (rows only grow along
// a warp's sequence).
__device__ __forceinline__ int next_problem(const int64_t *__restrict__ begin, int count, int q,
                                            int64_t x)
{
    if (q + 1 >= count || begin[q + 1] > x) return q;
    return find_problem(begin, count, x);
}

enum { MODE_COUNT = 0, MODE_EMIT = 1, MODE_FUSED = 2 };

struct WalkArgs {
    const BatchIndex *B;
    int warp_smem;           // shared-memory bytes of one warp
    int row_block;           // rows a warp claims per atomic
    int rec_max;             // bytes of one record buffer
    int64_t *row_ptr;        // COUNT: per-row counts; FUSED: row pointers; EMIT: read
    int32_t *col;
    float *lo, *up;
    float4 *acc;             // COUNT: the row's FP32 sums, for terms_fp32
    double *trunc;           // FUSED: outside-window mass in, full truncated mass out
    double *sink_lo, *sink_up;
    uint32_t *flags;
    uint32_t *status;        // [0] status bits, [1] look-back abort flag
    unsigned long long *lb;  // FUSED: look-back words, zeroed, one per row
    int64_t capacity;        // pairs the output arrays hold (< 0: unchecked)
    int64_t total_at;        // EMIT: index of the total in row_ptr
    int spin_limit;          // look-back sleeps before giving up
    int64_t row_begin;       // the launch covers global rows [row_begin, row_end)
    int64_t row_end;
    int64_t stall_row;       // fault injection: this row never publishes (-1: none)
    int64_t fault_row;       // fault injection: this row's checks see a bad sum (-1: none)
    int64_t guard_row;       // fault injection: this row reports a damaged record (-1: none)
};

// A dimension's entry as finish_dim makes it: the window within the record's
// tables, chunks of whole parents within a list, the division by its width.
__device__ __forceinline__ bool sound_dim(const RecDim &h, int lay, int tsum_cap)
{
    const bool narrow = (unsigned)(h.tw - 1) < 32u;
    return (narrow ? (unsigned)((lay >> 16) - 33) < 32u : lay == 0) &&
           (unsigned)h.tw <= (unsigned)tsum_cap && (unsigned)h.tb <= (unsigned)(tsum_cap - h.tw) &&
           (h.tw == 0 || (uint32_t)h.tw * h.magic < (uint32_t)h.tw);
}

// SAVED (an emit): the records have lain in the caller's workspace since the
// count. Every row's are checked before it is walked: widths, chunks and
// addresses out of a record that was overwritten would take the walk out of its
// lists or keep it going for ever. (In every emit the check would cost the 7-D
// building 0.03 of 4.50 ms.)
template <int MODE, bool SAVED>
__global__ void __launch_bounds__(IMPACT_TREE_WARPS_MAX * 32, 4) walk_fp32(const WalkArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool kCount = MODE != MODE_EMIT;
    constexpr bool kEmit = MODE != MODE_COUNT;
    const int lane = threadIdx.x & 31;
    unsigned char *const wbase = smem_raw + (size_t)(threadIdx.x >> 5) * A.warp_smem;
    const BatchIndex *B = A.B;
    if (MODE == MODE_EMIT && A.capacity >= 0 && A.row_ptr[A.total_at] > A.capacity) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(A.status, IMPACT_STATUS_CAPACITY);
        return;
    }
    unsigned long long *const next_row = B->next_row + (MODE == MODE_EMIT ? 1 : 0);

    // persistent: each warp takes rows from the batch's row counter,
    // A.row_block consecutive rows per atomic (one counter serves every warp
    // of the grid: claiming short rows one by one queues the atomics), in
    // ascending order. The count pass takes
    // rows one ahead: while a warp walks a row, the next row's record is copied
    // (cp.async) into the warp's other record buffer. The emit pass (more
    // registers live in its walk) copies each record when it starts it. So does the
    // one-pass walk, one row at a time: a row taken and not yet counted holds up
    // every row after it while its warp waits for the rows before the one it is at
    // (a row ahead: the 11^5 room 85 ms, the unicycle 139; none: 14.1 and 22.4).
    constexpr bool kAhead = MODE == MODE_COUNT;
    const int64_t row_end = A.row_end;
    unsigned char *const work = wbase + (kAhead ? 2 : 1) * A.rec_max;
    // the claimed rows [claim[0], claim[1]) stand in the last bytes of the
    // warp's block (not in registers: the walk needs all of them)
    unsigned long long *const claim =
        reinterpret_cast<unsigned long long *>(wbase + A.warp_smem - kClaimBytes);
    if (lane == 0) claim[0] = claim[1] = 0;
    __syncwarp();
    auto take = [&]() -> int64_t {
        unsigned long long t = claim[0];
        if (t == claim[1]) {   // warp-uniform: every lane reads the same words
            unsigned long long c = 0;
            if (lane == 0) c = atomicAdd(next_row, (unsigned long long)A.row_block);
            t = __shfl_sync(0xffffffffu, c, 0);
            if (lane == 0) claim[1] = t + A.row_block;
        }
        __syncwarp();
        if (lane == 0) claim[0] = t + 1;
        __syncwarp();
        return A.row_begin + (int64_t)t;
    };
    auto fetch = [&](int64_t row, int &q, unsigned char *dst) {
        if (row >= row_end) return;
        q = next_problem(B->row_begin, B->count, q, row);
        const ImpactDesc &D = *B->desc[q];
        const int stride = D.rec_stride;
        const unsigned char *src = B->rec[q] + (row - B->row_begin[q]) * (int64_t)stride;
        // a count with a shared leaf table reads no table of the last two
        // dimensions
        const int bytes = MODE == MODE_COUNT && D.leaf_shared
                              ? (int)(sizeof(RecDim) * D.n + sizeof(RecRow)) + 8 * D.dim[D.n - 2].rec_off
                              : stride;
        for (int i = lane; i < (bytes >> 4); i += 32) cp_async16(dst + 16 * i, src + 16 * i);
    };
    int64_t row = take();
    int q = 0, b = 0;
    if (kAhead) {
        fetch(row, q, wbase);
        cp_async_commit();
    }
    while (row < row_end) {
        int64_t nxt = 0;
        int q_nxt = q;
        if (kAhead) {
            nxt = take();
            fetch(nxt, q_nxt, wbase + (b ^ 1) * A.rec_max);
            cp_async_commit();
            cp_async_wait_prior();   // this row's record has landed
        } else {
            fetch(row, q, wbase);
            cp_async_commit();
            cp_async_wait_all();
        }
        __syncwarp();
        const ImpactDesc &D = *B->desc[q];
        const int n = D.n;
        const float cut = D.cutoff32;
        unsigned char *const rec = wbase + b * A.rec_max;
        const WarpMem S = carve(work, rec, n, D.leaf_cap);
        const bool empty = __any_sync(0xffffffffu, lane < n && S.h[lane].tw == 0);
        bool walked = true;
        if (SAVED)   // fault injection: as if the record's chunks were overwritten
            walked = !__any_sync(0xffffffffu,
                                 lane < n && !sound_dim(S.h[lane],
                                                        row == A.guard_row ? 1 : S.h[lane].lay,
                                                        D.tsum_cap)) &&
                     (!D.lists || (uint64_t)rec_row(rec, n)->leaf < (uint64_t)D.leaf_items);
        else if (kCount)
            walked = row != A.guard_row;
        Leaf f = leaf_of(S, n);
        bool lb_ok = true;
        int64_t base = 0, len = 0;
        if (kCount) {
            CountAcc acc;
            if (!empty && walked) {
                if (MODE == MODE_COUNT && D.leaf_shared) {
                    const unsigned char *tab = B->leaf[q] + rec_row(rec, n)->leaf * D.leaf_stride;
                    if (reinterpret_cast<const LeafHead *>(tab)->nb > 0) {
                        f.shared = reinterpret_cast<const float4 *>(tab + sizeof(LeafHead));
                    } else {   // too wide for a table: the last two windows after all
                        const unsigned char *src = B->rec[q] + (row - B->row_begin[q]) * (int64_t)D.rec_stride;
                        const int from = (int)(sizeof(RecDim) * n + sizeof(RecRow)) + 8 * D.dim[n - 2].rec_off;
                        for (int i = (from >> 4) + lane; i < (D.rec_stride >> 4); i += 32)
                            cp_async16(rec + 16 * i, src + 16 * i);
                        cp_async_commit();
                        cp_async_wait_all();
                        __syncwarp();
                    }
                }
                if (!f.shared) leaf_build(S, n, f, lane, cut);
                if (MODE == MODE_FUSED) {
                    int none = 0;
                    walk_row<true>(S, n, f, false, 0, lane, acc, EmitOut{}, none, cut);
                } else {
                    count_row(S, n, f, lane, acc, cut);
                }
            }
            const int c = __reduce_add_sync(0xffffffffu, acc.cnt);
            const float drop = warp_sum_ru(acc.drop);
            const float sup = warp_sum_ru(acc.sup);
            const float slo = warp_sum_rd(acc.slo);
            if (MODE == MODE_FUSED) {
                int64_t prefix = 0;
                lb_ok = lookback(A.lb, row, c, lane, A.status + 1, A.status, A.spin_limit,
                                 row == A.stall_row, prefix);
                if (lane == 0 && lb_ok) {
                    A.row_ptr[row] = prefix;
                    if (row == B->rows - 1) {   // the total, also beside the status
                        A.row_ptr[B->rows] = prefix + c;
                        reinterpret_cast<int64_t *>(A.status)[1] = prefix + c;
                    }
                }
                base = prefix;
                len = c;
                if (lane == 0) {
                    // FP64 row terms: the dropped in-window mass joins the mass
                    // outside the window box; then the row checks of Def. 3.1
                    const double tr = __dadd_ru(A.trunc[row], (double)drop);
                    A.trunc[row] = tr;
                    if (A.flags) {
                        const double slv = A.sink_lo[row], suv = A.sink_up[row];
                        const double lo_sum = row == A.fault_row ? 2.0 : (double)slo;
                        uint32_t fl = 0;
                        if (__dadd_rd(lo_sum, slv) > 1.0) fl |= IMPACT_ROW_LO_SUM_ABOVE_ONE;
                        if (__dadd_ru(__dadd_ru((double)sup, suv), tr) < 1.0)
                            fl |= IMPACT_ROW_UP_SUM_BELOW_ONE;
                        A.flags[row] = fl;
                        if (fl) atomicOr(A.status, IMPACT_STATUS_UNSOUND);
                    }
                }
            } else if (lane == 0) {
                A.row_ptr[row] = c;   // counts; the scan turns them into row pointers
                A.acc[row] = make_float4(drop, sup, slo, 0.0f);   // terms_fp32 finishes the row
            }
        } else {
            base = A.row_ptr[row];
            len = A.row_ptr[row + 1] - base;
        }
        if (kEmit && walked && lb_ok) {
            if (base < 0 || len < 0 || (A.capacity >= 0 && base + len > A.capacity)) {
                if (lane == 0)
                    atomicOr(A.status, MODE == MODE_FUSED ? IMPACT_STATUS_CAPACITY
                                                          : IMPACT_STATUS_EMIT_MISMATCH);
            } else {
                const EmitOut out{A.col + base, A.lo + base, A.up + base, (int)len};
                int written = 0;
                __syncwarp();   // FUSED: the count's leaf table makes room
                if (!empty) {
                    // the row's list block, where the build shares leaf tables
                    const bool lists = MODE == MODE_EMIT && D.lists && f.nb >= kListMin &&
                                       f.nb <= kListMax;
                    const int after = emit_leaf_bytes(D.leaf_cap, true) - kInfoBytes - 4 * kStartWords;
                    if (lists) {
                        const unsigned char *src = B->leaf[q] +
                                                   rec_row(rec, n)->leaf * D.leaf_stride +
                                                   leaf_lists_at(D.leaf_cap);
                        unsigned char *dst = reinterpret_cast<unsigned char *>(S.leaf);
                        for (int i = lane; i < (list_block(f.nb) >> 4); i += 32)
                            cp_async16(dst + 16 * i, src + 16 * i);
                        cp_async_commit();
                        cp_async_wait_all();
                        __syncwarp();
                    }
                    CountAcc none;
                    walk_row<false>(S, n, f, lists, after, lane, none, out, written, cut);
                }
                if (lane == 0 && written != len) atomicOr(A.status, IMPACT_STATUS_EMIT_MISMATCH);
            }
        }
        if (lane == 0 && !walked) atomicOr(A.status, IMPACT_STATUS_INTERNAL);
        if (!lb_ok) break;   // the rows after this one cannot find their offsets
        __syncwarp();        // every lane is done with the buffer before it is refilled
        if (kAhead) {
            row = nxt;
            q = q_nxt;
            b ^= 1;
        } else {
            row = take();
        }
    }
    cp_async_wait_all();
}

int occupancy_grid(const void *kernel, int threads, size_t smem, int64_t work_items,
                   int items_per_block)
{
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem);
    if (occ < 1) occ = 1;
    int64_t want = (work_items + items_per_block - 1) / items_per_block;
    int64_t cap = (int64_t)sms * occ;
    return (int)std::max<int64_t>(1, std::min(want, cap));
}

}  // namespace

namespace impact {

int64_t record_stride(int n, int tsum_cap)
{
    return ((int64_t)32 * n + 16 + (int64_t)8 * tsum_cap + 15) / 16 * 16;
}

int walk_work_bytes(const ImpactDesc &D, int mode)
{
    // rows with a shared leaf table stage none of their own to count, and
    // rows of at most two dimensions none at all
    const int emit = D.n > 2 ? emit_leaf_bytes(D.leaf_cap, mode == MODE_EMIT && D.lists) : 0;
    const int count = D.n > 2 || !(D.cutoff32 > 0.0f) ? 32 * (D.leaf_cap + 1) : 0;
    if (mode == MODE_EMIT) return list_bytes(D.n) + align16(emit);
    if (mode == MODE_COUNT) return list_bytes(D.n) + align16(D.leaf_shared ? 0 : count);
    return list_bytes(D.n) + align16(emit > count ? emit : count);
}

int walk_core_bytes(int n, int tsum_cap, int leaf_cap)
{
    const int64_t b = 2 * record_stride(n, tsum_cap) + list_bytes(n) + align16(32 * (leaf_cap + 1));
    return (int)std::min<int64_t>(b, INT32_MAX / 2);
}

// Windows by groups of lanes (setup_dim_split) while they leave the chip idle. One
// lane each against groups: items_fp32 22.6 against 10.8 us (robot 21^2, 4k rows),
// 13.1 against 10.4 (room 9^5, 11k items), 14.1 against 16.3 (room 11^5, 20k);
// per row 18.5 against 12.0 us (33x31 cells, 4 inputs, 256 units), 16.6 against
// 11.5 (9^3, 292), 18.1 against 24.0 (64^2, 1024), 48.7 against 119 (160^2, 6400).
constexpr int64_t kSplitItems = 12288;
constexpr int64_t kSplitUnits = 456;   // three warps of setup_fp32 per SM

// Shared windows pay when a window serves three rows or more (below that the
// items' write and read back cost about what they save): the 11^5 room's 20k
// windows take 0.014 ms and the gather of 1.45M records 0.37 ms, one setup per
// row 1.39 ms; building 6^7 0.44 against 1.79 ms. Leaf tables pay when one
// serves four rows or more and all of them take less than the records: the
// unicycle 51x51x25 (26k tables of about 200 entries for 1.3M rows) sorted them
// per row in 11.7 ms of count pass, and takes 0.28 ms for the tables and 1.1 ms
// for the pass.
void size_items32(ImpactDesc &D, int64_t &item_bytes, int64_t &leaf_bytes)
{
    const int n = D.n;
    int64_t bytes = 0, items = 0;
    for (int d = 0; d < n; ++d) {
        ImpactDim &g = D.dim[d];
        g.item_stride = (int)sizeof(DimOut) + 8 * ((g.wcap + 1) & ~1);
        g.item_off = bytes;
        bytes += g.n_items * (int64_t)g.item_stride;
        items += g.n_items;
    }
    D.share32 = D.kind != KIND_IMAGES && items * 3 <= D.rows * n;
    item_bytes = D.share32 ? bytes : 0;
    for (int d = 0; d < n; ++d) D.dim[d].group = items <= kSplitItems ? 8 : 1;
    const bool lists = D.leaf_cap >= kListCapMin && D.leaf_cap <= kListCapMax;
    D.leaf_stride = leaf_lists_at(D.leaf_cap) + (lists ? list_block(kListMax) : 0);
    D.leaf_shared = D.share32 && n >= 3 && D.cutoff32 > 0.0f && D.leaf_items * 4 <= D.rows &&
                    D.leaf_items * D.leaf_stride <= D.rows * (int64_t)D.rec_stride;
    D.lists = D.leaf_shared && lists;
    leaf_bytes = D.leaf_shared ? D.leaf_items * D.leaf_stride : 0;
}

int leaf32_bytes(const ImpactDesc &D)
{
    const int w = ((D.dim[D.n - 2].wcap + 1) & ~1) + ((D.dim[D.n - 1].wcap + 1) & ~1);
    return 2 * (int)sizeof(RecDim) + 8 * w + align16(32 * (D.leaf_cap + 1)) +
           (D.lists ? list_block(kListMax) : 0);
}

cudaError_t launch_setup_fp32(const BatchIndex *d_index, int64_t units, bool shared, bool own,
                              int64_t item_units, uint32_t *status, cudaStream_t stream)
{
    if (units <= 0) return cudaSuccess;
    if (own && units <= kSplitUnits) {
        const int g = occupancy_grid((const void *)setup_split_fp32, 128, 0, units * 6, 128 / 32);
        setup_split_fp32<<<g, 128, 0, stream>>>(d_index, status);
    } else if (own) {
        const int g = occupancy_grid((const void *)setup_fp32, 256, 0, units, 256 / 32);
        setup_fp32<<<g, 256, 0, stream>>>(d_index, status);
    }
    if (shared) {
        const int gi = occupancy_grid((const void *)items_fp32, 128, 0, item_units, 128 / 32);
        items_fp32<<<gi, 128, 0, stream>>>(d_index, status);
        const int gr = occupancy_grid((const void *)rows_fp32, 256, 0, units, 256 / 32);
        rows_fp32<<<gr, 256, 0, stream>>>(d_index);
    }
    return cudaGetLastError();
}

cudaError_t launch_terms_fp32(const BatchIndex *d_index, int64_t rows, const void *acc,
                              int64_t fault_row, const RowOutputs &o, const ScanHead &scan,
                              cudaStream_t stream)
{
    if (rows <= 0) return cudaSuccess;
    const int g = occupancy_grid((const void *)terms_fp32, kTermThreads, 0, rows, kTermThreads);
    terms_fp32<<<scan.tiles + g, kTermThreads, 0, stream>>>(
        d_index, (const float4 *)acc, fault_row, o.sink_lo, o.sink_up, o.trunc, o.flags, o.status,
        scan);
    return cudaGetLastError();
}

cudaError_t launch_leaf_fp32(const BatchIndex *d_index, int64_t tables, int leaf_smem,
                             cudaStream_t stream)
{
    if (tables <= 0) return cudaSuccess;
    const size_t smem = (size_t)leaf_smem * 4;
    cudaError_t e = allow_smem((const void *)leaf_fp32);
    if (e != cudaSuccess) return e;
    const int g = occupancy_grid((const void *)leaf_fp32, 128, smem, tables, 4);
    leaf_fp32<<<g, 128, smem, stream>>>(d_index, leaf_smem);
    return cudaGetLastError();
}

cudaError_t launch_walk_fp32(const BatchIndex *d_index, int64_t row_begin, int64_t row_end,
                             int rec_max, const int work_max[3], int warps, int mode,
                             bool saved, const RowOutputs &o,
                             unsigned long long *lb, const WalkFaults &f, cudaStream_t stream)
{
    const int64_t rows = row_end - row_begin;
    if (rows <= 0) return cudaSuccess;
    // record buffers and warp blocks start 16-byte aligned (record strides are
    // multiples of 16)
    rec_max = (rec_max + 15) & ~15;
    const int work = work_max[mode];
    const int warp_smem = (mode == MODE_COUNT ? 2 : 1) * rec_max + ((work + 15) & ~15) + kClaimBytes;
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    warps = std::max(1, std::min({warps, IMPACT_TREE_WARPS_MAX, optin / std::max(warp_smem, 1)}));
    const int threads = warps * 32;
    const size_t smem = (size_t)warp_smem * warps;
    auto kernel = mode == MODE_COUNT   ? walk_fp32<MODE_COUNT, false>
                  : mode == MODE_FUSED ? walk_fp32<MODE_FUSED, false>
                  : saved              ? walk_fp32<MODE_EMIT, true>
                                       : walk_fp32<MODE_EMIT, false>;
    const void *k = (const void *)kernel;
    cudaError_t e = allow_smem(k);
    if (e != cudaSuccess) return e;
    WalkArgs A;
    A.B = d_index;
    A.warp_smem = warp_smem;
    A.rec_max = rec_max;
    A.row_ptr = o.row_ptr;
    A.col = o.col;
    A.lo = (float *)o.lo;
    A.up = (float *)o.up;
    A.acc = (float4 *)lb;
    A.trunc = o.trunc;
    A.sink_lo = o.sink_lo;
    A.sink_up = o.sink_up;
    A.flags = o.flags;
    A.status = o.status;
    A.lb = lb;
    A.capacity = o.capacity;
    A.total_at = o.total_at;
    A.spin_limit = f.spin_limit > 0 ? f.spin_limit : (1 << 24);
    A.row_begin = row_begin;
    A.row_end = row_end;
    A.stall_row = f.stall_row;
    A.fault_row = f.fault_row;
    A.guard_row = f.guard_row;
    // persistent grid: as many blocks as fit at once (rows are taken dynamically)
    const int g = occupancy_grid(k, threads, smem, rows, warps);
    // rows per claim: 4 in the count pass (its rows are short: the atomics
    // cost more than the last claims' imbalance), in the emit up to 4 while that
    // imbalance (up to 3 rows per warp) stays under 1/256 of each warp's rows
    A.row_block = mode == MODE_COUNT   ? 4
                  : mode == MODE_FUSED ? 1
                      : (int)std::max<int64_t>(
                            1, std::min<int64_t>(4, rows / ((int64_t)g * warps * 256)));
    kernel<<<g, threads, smem, stream>>>(A);
    return cudaGetLastError();
}

}  // namespace impact
