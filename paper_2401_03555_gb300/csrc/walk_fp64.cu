// walk_fp64.cu -- FP64-plain construction (Def. 3.1, Sec. 4.4 cutoff, Remark
// 4.1 sink) in three steps. Every value is that of the definition in FP64
// round-to-nearest, factors multiplied in the order of the dimensions.
//
//   items_fp64  the factor tables of every distinct image (impact_desc.h:
//               rows that read the same coordinates and offset share an
//               item). A group of 8, 16 or 32 lanes makes one item, one lane
//               per window edge: erfc once per edge and image end, the masses
//               of the cells between from neighbouring lanes; then the trimmed
//               window, its sums and, for the last dimension, the targets
//               sorted by upper factor with prefix sums.
//   walk_fp64   one warp per row: the prefix tree of target cells level by
//               level in C order over the dimensions but the last, as in the
//               FP32 walk; a node is dropped when even the largest later
//               factors cannot lift it to the cutoff. The count pass finds how
//               many targets of the last dimension pass under each parent by a
//               search in the sorted table (RN(P u) is monotone in u), the
//               emit pass tests every target under every parent, one lane each.
//   terms_fp64  after the count, one thread per row: sink bounds, truncated mass
//               and row checks.
//
// What bounds it: FP64 issue (2 lanes per clock and SM on this part, so a
// warp-wide multiply holds the pipe 16 clocks) and the 20 bytes a pair writes.
// erfc costs about a hundred FP64 instructions: evaluated per pair and
// dimension it was the whole run time, per image and edge it is little. Whole
// builds, per-pair kernel -> this one: unicycle 21x19x13 (25.6M pairs) 395 ->
// 0.56 ms (items 0.05, count 0.22, emit 0.22), room 5x6x5x6x5 303 -> 0.37 ms,
// dense robot 21x21 14.0 -> 0.27 ms (host-bound). Both walks keep the FP64 pipe
// 80% busy, so what is not a product stays off it: compares on bits, FP32
// searches, no conversions.
#include <cuda_runtime.h>
#include <float.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "impact_desc.h"
#include "kernels.h"
#include "launch.h"
#include "rowmath.cuh"
#include "scan.cuh"

namespace {

using namespace rowmath;

constexpr int kCap = 64;              // nodes per level list (one chunk)
constexpr int kSortMax = 256;         // widest last-dimension window that is sorted
constexpr int kTablesMax = 2048;      // widest window box (targets, all dimensions)
constexpr int kWarps = 8;             // warps per block at most
constexpr int kSmemWarp = 64 * 1024;  // shared memory of one warp at most
constexpr int64_t kItemsMax = (int64_t)1 << 30;   // item tables of one build at most

// One item: the header, the window's (U, L) pairs and, in the last dimension
// of a build with a cutoff, five sorted arrays of w64 + 1 doubles (su, sl, pu,
// pl, sf: upper factors descending with their lower factors, prefix sums of
// both, suffix sums of su).
struct Item64 {
    double SW;             // sum of U over the trimmed window
    double O;              // mass outside the trimmed window
    double gmax, gmin;     // in-domain mass: largest, smallest over the image
    float M32;             // largest U of the trimmed window, rounded up
    int ta, tw;            // trimmed window [ta, ta + tw)
    int first;             // its first entry in the table
};
static_assert(sizeof(Item64) == 48, "Item64 layout");
constexpr int kItemHead = 64;

__host__ __device__ inline bool is_sorted_dim(float cutoff32, int w64)
{
    return cutoff32 > 0.0f && w64 <= kSortMax;
}

__device__ __forceinline__ double2 *item_table(unsigned char *it)
{
    return reinterpret_cast<double2 *>(it + kItemHead);
}

__device__ __forceinline__ double *item_sorted(unsigned char *it, int w64)
{
    return reinterpret_cast<double *>(it + kItemHead + 16 * (int64_t)w64);
}

__device__ __forceinline__ double group_sum(unsigned mask, double v, int G)
{
    for (int o = G >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o, G);
    return v;
}

__device__ __forceinline__ double group_scan(unsigned mask, double v, int sub, int G)
{
    for (int o = 1; o < G; o <<= 1) {
        const double y = __shfl_up_sync(mask, v, o, G);
        if (sub >= o) v += y;
    }
    return v;
}

// Item tables. A warp unit is 32 / group items of one dimension of one build;
// the loops over a window run to the warp's widest, so its groups stay together
// (to the dimension's, caller images paid for the whole grid: 20,000 of 1000 cells
// with windows of 20 took 5.8 ms a build).
__global__ void __launch_bounds__(256)
items_fp64(const BatchIndex *__restrict__ B, uint32_t *__restrict__ status)
{
    const unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = warp0; u < B->item_units; u += nwarps) {
        const int seg = find_problem(B->item_begin, B->count * IMPACT_MAX_DIM, u);
        const int q = seg / IMPACT_MAX_DIM, d = seg % IMPACT_MAX_DIM;
        const ImpactDesc &D = *B->desc[q];
        const ImpactDim &g = D.dim[d];
        const int G = g.group, sub = lane % G;
        const int64_t c = (u - B->item_begin[seg]) * (32 / G) + lane / G;
        const bool act = c < g.n_items;
        const int64_t cc = act ? c : 0;   // idle groups repeat item 0 and store nothing
        unsigned char *it = B->items[q] + g.item_off + cc * g.item_stride;
        double2 *ul = item_table(it);
        const double *E = D.edges + g.edge_off;
        double mlo, mhi;
        {
            int idx[IMPACT_MAX_DIM], j = 0;
            if (D.kind != KIND_IMAGES) decode_item(D, d, cc, idx, j);
            image_dim<false>(D, cc, idx, j, d, mlo, mhi);
        }
        int a, b;
        window_dim(g, mlo, mhi, a, b);
        int W = b - a + 1;
        if (W > g.w64) {   // cannot happen for the planner's bound
            if (act && sub == 0) atomicOr(status, IMPACT_STATUS_TABLE_OVERFLOW);
            W = g.w64;
            b = a + W - 1;
        }
        const double cut = D.cutoff, inv_s = g.inv_s;
        // targets k0 .. k0 + G - 2 per step: lane `sub` takes edge k0 + sub,
        // and the last lane only lends its edge to the one before it. The
        // arguments that no edge gives (the domain's edges at both image ends,
        // slots 0-3, and at its clamped midpoint, 4-5; targets whose midpoint
        // lies in the image, two each) share a round of erfc of their own,
        // one per lane: a warp-wide erfc costs the same for one lane as for 32
        int first = INT_MAX, last = -1;
        const int shift = lane - sub;
        const unsigned gmask = G == 32 ? kAll : (1u << G) - 1u;
        double tx = 0.0, tf = 0.0;             // slots 0-5, in lanes 0-5
        double ax = 0.0, af = 0.0;             // edge a at m_lo, in lane 0
        double wx = 0.0, wf = 0.0;             // edge a + W at m_hi, in lane wlane
        int wlane = 0;
        // the warp's widest window (an empty one has an edge too)
        const int edges = max(__reduce_max_sync(kAll, W), 1);
        for (int k0 = 0; k0 < edges; k0 += G - 1) {
            const int k = k0 + sub;
            const double c0 = E[min(a + k, g.N)];
            const double x0 = (c0 - mlo) * inv_s, x1 = (c0 - mhi) * inv_s;
            const double f0 = erfc(fabs(x0)), f1 = erfc(fabs(x1));
            if (k0 == 0) {
                ax = x0;
                af = f0;
            }
            const unsigned at_w = (__ballot_sync(kAll, k == W) >> shift) & gmask;
            if (at_w) wlane = __ffs(at_w) - 1;
            if (k == W) {
                wx = x1;
                wf = f1;
            }
            const double e0 = __shfl_down_sync(kAll, c0, 1, G);
            const double y0 = __shfl_down_sync(kAll, x0, 1, G), y1 = __shfl_down_sync(kAll, x1, 1, G);
            const double h0 = __shfl_down_sync(kAll, f0, 1, G), h1 = __shfl_down_sync(kAll, f1, 1, G);
            const bool mine = sub < G - 1 && k < W;
            const double mid = 0.5 * (c0 + e0);
            const bool inner = mine && !(mid < mlo) && !(mid > mhi);
            const unsigned inners = (__ballot_sync(kAll, inner) >> shift) & gmask;
            const int base = k0 == 0 ? 6 : 0, slots = base + 2 * __popc(inners);
            const int my_slot = base + 2 * __popc(inners & ((1u << sub) - 1u));
            const int most = __reduce_max_sync(kAll, slots);
            double qa = 0.0, qfa = 0.0, qb = 0.0, qfb = 0.0;
            for (int s0 = 0; s0 < most; s0 += G) {
                const int s = s0 + sub;
                double x = 0.0, f = 0.0;
                if (s < slots) {
                    double edge, m;
                    if (s < base) {
                        edge = s & 1 ? g.hi : g.lo;
                        m = s < 2 ? mlo : s < 4 ? mhi : clampd(0.5 * (g.lo + g.hi), mlo, mhi);
                    } else {
                        unsigned rest = inners;
                        for (int r = (s - base) >> 1; r > 0; --r) rest &= rest - 1;
                        const int kk = a + k0 + __ffs(rest) - 1;
                        m = 0.5 * (E[kk] + E[kk + 1]);
                        edge = E[kk + ((s - base) & 1)];
                    }
                    x = (edge - m) * inv_s;
                    f = erfc(fabs(x));
                }
                if (base > 0 && s0 == 0) {
                    tx = x;
                    tf = f;
                }
                const int src = my_slot & (G - 1);
                const double xa = __shfl_sync(kAll, x, src, G), fa = __shfl_sync(kAll, f, src, G);
                const double xb = __shfl_sync(kAll, x, src + 1, G), fb = __shfl_sync(kAll, f, src + 1, G);
                if (my_slot >= s0 && my_slot < s0 + G) {
                    qa = xa;
                    qfa = fa;
                    qb = xb;
                    qfb = fb;
                }
            }
            if (mine) {
                const double glo = mass64(x0, f0, y0, h0), ghi = mass64(x1, f1, y1, h1);
                // largest factor: at the midpoint clamped to the image
                const double U = mid < mlo ? glo : mid > mhi ? ghi : mass64(qa, qfa, qb, qfb);
                if (act) ul[k] = make_double2(U, fmin(glo, ghi));
                if (U >= cut) {
                    first = min(first, k);
                    last = k;
                }
            }
        }
        for (int o = G >> 1; o > 0; o >>= 1) {
            first = min(first, __shfl_xor_sync(kAll, first, o, G));
            last = max(last, __shfl_xor_sync(kAll, last, o, G));
        }
        __syncwarp();
        const bool empty = last < 0;
        double sw = 0.0, ow = 0.0, M = 0.0;
        for (int k = sub; act && k < W; k += G) {
            const double v = ul[k].x;
            if (!empty && k >= first && k <= last) {
                sw += v;
                M = fmax(M, v);
            } else {
                ow += v;
            }
        }
        // the masses beyond the window at m_lo and m_hi and in the domain at
        // its clamped midpoint, m_lo and m_hi, one per lane
        const int sa = sub == 2 ? 4 : sub == 4 ? 2 : 0, sb = sub == 2 ? 5 : sub == 3 ? 1 : 3;
        double pa = __shfl_sync(kAll, tx, sa, G), fa = __shfl_sync(kAll, tf, sa, G);
        double pb = __shfl_sync(kAll, tx, sb, G), fb = __shfl_sync(kAll, tf, sb, G);
        const double qx = __shfl_sync(kAll, wx, wlane, G), qf = __shfl_sync(kAll, wf, wlane, G);
        if (sub == 0) {
            pb = ax;
            fb = af;
        } else if (sub == 1) {
            pa = qx;
            fa = qf;
        }
        double part = 0.0;
        if (sub == 0 ? a > 0 : sub == 1 ? b < g.N - 1 : sub < 5) part = mass64(pa, fa, pb, fb);
        sw = group_sum(kAll, sw, G);
        ow = group_sum(kAll, ow, G);
        for (int o = G >> 1; o > 0; o >>= 1) M = fmax(M, __shfl_xor_sync(kAll, M, o, G));
        const double left = __shfl_sync(kAll, part, 0, G), right = __shfl_sync(kAll, part, 1, G);
        const double gmax = __shfl_sync(kAll, part, 2, G);
        const double gmin = fmin(__shfl_sync(kAll, part, 3, G), __shfl_sync(kAll, part, 4, G));
        const int tw = empty ? 0 : last - first + 1;
        if (act && sub == 0) {
            Item64 h;
            h.SW = sw;
            h.O = ow + left + right;
            h.gmax = gmax;
            h.gmin = gmin;
            h.M32 = __double2float_ru(M);
            h.ta = empty ? a : a + first;
            h.tw = tw;
            h.first = empty ? 0 : first;
            *reinterpret_cast<Item64 *>(it) = h;
        }
        if (d != D.n - 1 || !is_sorted_dim(D.cutoff32, g.w64)) continue;   // uniform in the warp
        const int cs = g.w64 + 1;
        double *su = item_sorted(it, g.w64), *sl = su + cs, *pu = sl + cs, *pl = pu + cs, *sf = pl + cs;
        for (int k = sub; act && k < tw; k += G) {
            const double2 v = ul[first + k];
            int r = 0;
            for (int i = 0; i < tw; ++i) {
                const double x = ul[first + i].x;
                r += (x > v.x) || (x == v.x && i < k);
            }
            su[r] = v.x;
            sl[r] = v.y;
        }
        __syncwarp();
        double cu = 0.0, cl = 0.0, cf = 0.0;
        for (int k0 = 0; k0 < edges; k0 += G) {
            const int k = k0 + sub, kr = tw - 1 - k;   // forwards and from the end
            const bool in = act && k < tw;
            const double iu = group_scan(kAll, in ? su[k] : 0.0, sub, G) + cu;
            const double il = group_scan(kAll, in ? sl[k] : 0.0, sub, G) + cl;
            const double jf = group_scan(kAll, in ? su[kr] : 0.0, sub, G) + cf;
            if (in) {
                pu[k + 1] = iu;
                pl[k + 1] = il;
                sf[kr] = jf;
            }
            cu = __shfl_sync(kAll, iu, G - 1, G);
            cl = __shfl_sync(kAll, il, G - 1, G);
            cf = __shfl_sync(kAll, jf, G - 1, G);
        }
        if (act && sub == 0) {
            pu[0] = pl[0] = 0.0;
            sf[tw] = 0.0;
        }
    }
}

// Row terms after the count walk (acc: its dropped mass, upper and lower sums
// per row).
constexpr int kTermThreads = 256;
__global__ void __launch_bounds__(kTermThreads)
terms_fp64(const BatchIndex *__restrict__ B, const double *__restrict__ acc,
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
        if (!D.walk64) continue;
        const int64_t r = row - B->row_begin[q];
        int idx[IMPACT_MAX_DIM], j;
        decode_row(D, r, idx, j);
        // sink: 1 - prod of the in-domain masses. Outside the window box,
        // partitioned by the first dimension that leaves its window:
        // sum_k prod_{i<k} SW_i * O_k * prod_{i>k} (SW_i + O_i)
        double pmax = 1.0, pmin = 1.0, out = 0.0, pre = 1.0;
#pragma unroll
        for (int d = 0; d < IMPACT_MAX_DIM; ++d) {
            if (d < D.n) {
                const ImpactDim &g = D.dim[d];
                const Item64 *h = reinterpret_cast<const Item64 *>(
                    B->items[q] + g.item_off + item_of(D, r, idx, j, d) * g.item_stride);
                pmax *= h->gmax;
                pmin *= h->gmin;
                out = out * (h->SW + h->O) + pre * h->O;
                pre *= h->SW;
            }
        }
        const double sl = 1.0 - pmax, su = 1.0 - pmin, tr = out + acc[row];
        sink_lo[row] = sl;
        sink_up[row] = su;
        trunc[row] = tr;
        if (flags) {
            uint32_t f = 0;
            if (acc[2 * B->rows + row] + sl > 1.0 + 1e-12) f |= 0x1u;
            if (acc[B->rows + row] + su + tr < 1.0 - 1e-12) f |= 0x2u;
            flags[row] = f;
            if (f) atomicOr(status, IMPACT_STATUS_UNSOUND);
        }
    }
}

// ---------------------------------------------------------------------------
// the walk
// ---------------------------------------------------------------------------

// Per (row, dimension) numbers of the walk, in the warp's shared memory.
struct WalkDim {
    long long cp;      // bits of the least node product that can still reach the cutoff
    double SR;         // product of the later dimensions' window sums
    int tw;            // trimmed width
    int off;           // first entry in the warp's table
    int cb;            // column of the first target
    int stride;
    uint32_t magic;    // ceil(2^32 / tw) when tw > 1
    int pad;
};
static_assert(sizeof(WalkDim) == 40, "WalkDim layout");

__host__ __device__ inline int list_bytes64(int n) { return ((n - 1) * kCap * 20 + 15) & ~15; }

struct Warp64 {
    WalkDim *h;
    double2 *ul;
    double *su, *pu, *pl, *sf;   // the last dimension's sorted arrays (count pass)
    float *su32;                 // leading bits of su
    unsigned char *lists;
};

struct Nodes64 {
    double *P, *Pl;
    int *col;
};

__device__ __forceinline__ Nodes64 nodes(const Warp64 &S, int k)
{
    unsigned char *b = S.lists + k * (kCap * 20);
    Nodes64 L;
    L.P = reinterpret_cast<double *>(b);
    L.Pl = L.P + kCap;
    L.col = reinterpret_cast<int *>(L.Pl + kCap);
    return L;
}

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Sums of three values over the warp; lane k (k < 3) gets the k-th in x[0]. The
// lanes share the work (7 FP64 adds a lane and not 15: the pipe is busy 16
// clocks with each, whatever share of the lanes is active).
__device__ __forceinline__ void warp_sums(double (&x)[3], int lane)
{
    const unsigned m = 0xffffffffu;
    // halves keep (x0, x1) or (x2, -), quarters one of them each
    double a = lane & 16 ? x[2] : x[0], b = lane & 16 ? 0.0 : x[1];
    const double ga = lane & 16 ? x[0] : x[2], gb = lane & 16 ? x[1] : 0.0;
    a += __shfl_xor_sync(m, ga, 16);
    b += __shfl_xor_sync(m, gb, 16);
    double v = lane & 8 ? b : a;
    v += __shfl_xor_sync(m, lane & 8 ? a : b, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(m, v, o);
    // lanes 0, 8, 16 hold x0, x1, x2
    x[0] = __shfl_sync(m, v, (lane & 3) * 8);
}

struct Sums64 {
    int cnt = 0;
    double drop = 0.0, sup = 0.0, slo = 0.0;
};

struct Out64 {
    int32_t *col;
    double *lo, *up;
    int64_t len;
};

struct Node64 {
    double P, Pl;
    int c;
};

__device__ __forceinline__ Node64 node_at(const Nodes64 &L, bool root, int i)
{
    if (root) return Node64{1.0, 1.0, 0};
    return Node64{L.P[i], L.Pl[i], L.col[i]};
}

// The keep test x >= cut on the bits, which leaves the FP64 pipe to the products
// (a compare holds it as long as a multiply): the bits of non-negative doubles
// order like the doubles, and negative ones (a factor of rounded erfc
// differences can be a negative last bit) stay below; cutoff 0 keeps -0 too.
struct Cut64 {
    long long bits, also;   // keep iff bits(x) >= bits or bits(x) == also
    float sure, never;      // FP32 products from here on / below here decide (see search64)
};

// cut32: the smallest float that is not below cut.
__device__ __forceinline__ Cut64 cut_of(double cut, float cut32)
{
    Cut64 c;
    c.bits = __double_as_longlong(cut);
    c.also = cut32 > 0.0f ? c.bits : LLONG_MIN;
    // products below the normal range decide nothing
    const bool fine = cut32 > 1e-30f;
    c.sure = fine ? cut32 * 1.00001f : INFINITY;
    c.never = fine ? cut32 * 0.99999f : 0.0f;
    return c;
}

__device__ __forceinline__ bool passes(double x, const Cut64 &c)
{
    const long long b = __double_as_longlong(x);
    return b >= c.bits || b == c.also;
}

// A double's leading 24 bits as a float (rounded to zero; for values in the
// normal range of FP32 or 0, else some small or large float), without the FP64
// pipe's conversion.
__device__ __forceinline__ float lead32(double x)
{
    const long long b = __double_as_longlong(x);
    const int e = (int)(b >> 52);                       // sign and exponent
    const unsigned m = (unsigned)((unsigned long long)b >> 29);
    return e <= 896 ? 0.0f : __uint_as_float(m - (896u << 23));
}

// The bits of a non-negative float as a double (subnormals as 0).
__device__ __forceinline__ long long wide_bits(float x)
{
    const unsigned b = __float_as_uint(x);
    return b < (1u << 23) ? 0ll : ((long long)b << 29) + (896ll << 52);
}

// How many entries of su (descending) RN(P su) >= cut keeps: FP32 products of
// leading bits (within 2^-20 of the exact ones) decide all but those within
// 1e-5 of the cutoff, which take the FP64 product.
__device__ __forceinline__ int search64(double P, const double *su, const float *su32, int n,
                                        const Cut64 &cut)
{
    const float p = lead32(P);
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const float f = p * su32[mid];
        bool keep = f >= cut.sure;
        if (!keep && f >= cut.never) keep = __double_as_longlong(P * su[mid]) >= cut.bits;
        if (keep) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Children of candidates [c0, c1) of the level k - 1 list in dimension k, kept
// ones compacted into the level k list in order.
template <bool COUNT>
__device__ __forceinline__ int expand64(const Warp64 &S, int k, int c0, int c1, int lane,
                                        Sums64 &acc)
{
    const WalkDim h = S.h[k];
    const Nodes64 Lc = nodes(S, k), Lp = nodes(S, k > 0 ? k - 1 : 0);
    int nout = 0;
    for (int e0 = c0; e0 < c1; e0 += 32) {
        const int e = min(e0 + lane, c1 - 1);
        const bool act = e0 + lane < c1;
        const int pi = h.tw > 1 ? (int)__umulhi((uint32_t)e, h.magic) : e;
        const int t = e - pi * h.tw;
        const Node64 par = node_at(Lp, k == 0, pi);
        const double2 ul = S.ul[h.off + t];
        const double Pc = k > 0 ? par.P * ul.x : ul.x;
        const bool keep = act && __double_as_longlong(Pc) >= h.cp;
        if (COUNT && act && !keep) acc.drop += Pc * h.SR;
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (keep) {
            const int o = nout + __popc(bal & lanemask_lt());
            Lc.P[o] = Pc;
            Lc.Pl[o] = k > 0 ? par.Pl * ul.y : ul.y;
            Lc.col[o] = par.c + h.cb + t * h.stride;
        }
        nout += __popc(bal);
    }
    __syncwarp();
    return nout;
}

// The targets of the last dimension under npar parents, counted and summed.
__device__ __forceinline__ void leaf_count64(const Warp64 &S, int n, const Nodes64 &Lp, bool root,
                                             int npar, int lane, Sums64 &acc, const Cut64 &cut,
                                             bool sorted)
{
    const WalkDim h = S.h[n - 1];
    if (sorted) {
        for (int pi = lane; pi < npar; pi += 32) {
            const Node64 par = node_at(Lp, root, pi);
            const int lo = search64(par.P, S.su, S.su32, h.tw, cut);
            acc.cnt += lo;
            acc.sup += par.P * S.pu[lo];
            acc.slo += par.Pl * S.pl[lo];
            acc.drop += par.P * S.sf[lo];
        }
        return;
    }
    const int total = npar * h.tw;
    for (int e = lane; e < total; e += 32) {
        const int pi = h.tw > 1 ? (int)__umulhi((uint32_t)e, h.magic) : e;
        const Node64 par = node_at(Lp, root, pi);
        const double2 ul = S.ul[h.off + e - pi * h.tw];
        const double Pc = par.P * ul.x;
        if (passes(Pc, cut)) {
            acc.cnt += 1;
            acc.sup += Pc;
            acc.slo += par.Pl * ul.y;
        } else {
            acc.drop += Pc;
        }
    }
}

// The same targets, written: one lane per candidate, kept ones compacted.
__device__ __forceinline__ void leaf_emit64(const Warp64 &S, int n, const Nodes64 &Lp, bool root,
                                            int npar, int lane, const Out64 &out, int64_t &written,
                                            const Cut64 &cut)
{
    const WalkDim h = S.h[n - 1];
    const int total = npar * h.tw;
    for (int e0 = 0; e0 < total; e0 += 32) {
        const int e = min(e0 + lane, total - 1);
        const int pi = h.tw > 1 ? (int)__umulhi((uint32_t)e, h.magic) : e;
        const int t = e - pi * h.tw;
        const Node64 par = node_at(Lp, root, pi);
        const double2 ul = S.ul[h.off + t];
        const double Pc = par.P * ul.x;
        const bool keep = e0 + lane < total && passes(Pc, cut);
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        const int64_t p = written + __popc(bal & lanemask_lt());
        if (keep && p < out.len) {
            out.col[p] = par.c + h.cb + t;
            out.lo[p] = par.Pl * ul.y;
            out.up[p] = Pc;
        }
        written += __popc(bal);
    }
}

template <bool EMIT>
__device__ bool walk_row64(const Warp64 &S, int n, int lane, Sums64 &acc, const Out64 &out,
                           int64_t &written, const Cut64 &cut, bool sorted)
{
    auto leaves = [&](const Nodes64 &Lp, bool root, int npar) {
        if (EMIT) leaf_emit64(S, n, Lp, root, npar, lane, out, written, cut);
        else leaf_count64(S, n, Lp, root, npar, lane, acc, cut, sorted);
    };
    if (n == 1) {
        leaves(Nodes64{}, true, 1);
        return true;
    }
    const int last = n - 2;   // deepest list level
    // every step fills a list, leaves one or runs the leaves of one: bound
    // them by the candidates of every level (loose, overflow-safe)
    int64_t guard = 16, prod = 1;
    for (int k = 0; k <= last; ++k) {
        prod = min(prod * (int64_t)S.h[k].tw, (int64_t)1 << 40);
        guard += 8 * (int64_t)(k + 1) * (1 + prod / kCap);
    }
    int my_cur = 0, my_sz = 0;   // lane k: next candidate of level k, size of list k
    int k = 0;
    while (true) {
        if (--guard < 0) return false;
        if (k == last + 1) {
            leaves(nodes(S, last), false, __shfl_sync(0xffffffffu, my_sz, last));
            __syncwarp();   // the list is refilled next
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
        const int end = min(cur + kCap, total);
        const int nout = expand64<!EMIT>(S, k, cur, end, lane, acc);
        if (lane == k) {
            my_cur = end;
            my_sz = nout;
        }
        if (lane == k + 1) my_cur = 0;
        ++k;
    }
    return true;
}

struct Walk64Args {
    const BatchIndex *B;
    int warp_smem;
    int row_block;             // rows a warp claims per atomic
    int64_t *row_ptr;          // COUNT: per-row counts; EMIT: row pointers
    int32_t *col;
    double *lo, *up;
    double *acc;               // COUNT: [3][rows] dropped mass, upper and lower sums
    int64_t rows;
    uint32_t *status;
    int64_t capacity, total_at;
    int64_t row_begin, row_end;
    unsigned long long *next_row;
};

// Bytes of one warp's shared memory: per-dimension numbers, the row's trimmed
// tables, the last dimension's sorted arrays, the node lists.
__host__ __device__ inline int64_t warp_bytes64(int n, int64_t tsum, int wl, bool sorted)
{
    return 40 * n + (n & 1 ? 8 : 0) + 16 * tsum + (sorted ? 40 * (int64_t)((wl + 2) & ~1) : 0) +
           list_bytes64(n);
}

template <bool EMIT>
__global__ void __launch_bounds__(kWarps * 32) walk_fp64(const Walk64Args A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    unsigned char *const mine = smem + (size_t)(threadIdx.x >> 5) * A.warp_smem;
    const BatchIndex *B = A.B;
    if (EMIT && A.capacity >= 0 && A.row_ptr[A.total_at] > A.capacity) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(A.status, IMPACT_STATUS_CAPACITY);
        return;
    }
    const unsigned long long nrows = (unsigned long long)(A.row_end - A.row_begin);
    unsigned long long t = 0, t_end = 0;
    int q = 0;
    while (true) {
        if (t == t_end) {   // claim the next rows (ascending)
            unsigned long long c = 0;
            if (lane == 0) c = atomicAdd(A.next_row, (unsigned long long)A.row_block);
            t = __shfl_sync(0xffffffffu, c, 0);
            t_end = t + A.row_block;
        }
        if (t >= nrows) break;
        const int64_t row = A.row_begin + (int64_t)t;
        ++t;
        if (q + 1 < B->count && B->row_begin[q + 1] <= row) q = find_problem(B->row_begin, B->count, row);
        const ImpactDesc &D = *B->desc[q];
        if (!D.walk64) continue;
        const int n = D.n;
        const double cut = D.cutoff;
        const float cut32 = D.cutoff32;
        const Cut64 keep = cut_of(cut, cut32);
        const int64_t r = row - B->row_begin[q];
        const int wl = D.dim[n - 1].w64;
        const bool sorted = !EMIT && is_sorted_dim(cut32, wl);
        Warp64 S;
        S.h = reinterpret_cast<WalkDim *>(mine);
        S.ul = reinterpret_cast<double2 *>(mine + 40 * n + (n & 1 ? 8 : 0));
        // lane d: the item of dimension d
        unsigned char *it = nullptr;
        Item64 h;
        h.tw = 0;
        h.M32 = 1.0f;
        h.SW = 1.0;
        {
            int idx[IMPACT_MAX_DIM], j;
            decode_row(D, r, idx, j);
            if (lane < n) {
                const ImpactDim &g = D.dim[lane];
                it = B->items[q] + g.item_off + item_of(D, r, idx, j, lane) * g.item_stride;
                h = *reinterpret_cast<const Item64 *>(it);
            }
        }
        const bool empty = __any_sync(0xffffffffu, lane < n && h.tw == 0);
        int off = 0, tsum = 0;
        float R = 1.0f;
        double SR = 1.0;   // its products only where two factors meet
        for (int k = n - 1; k >= 0; --k) {
            const int twk = __shfl_sync(0xffffffffu, h.tw, k);
            const float Mk = __shfl_sync(0xffffffffu, h.M32, k);
            if (k < lane) off += twk;
            if (k > lane) R = __fmul_ru(R, Mk);
            tsum += twk;
            if (!EMIT) {
                const double SWk = __shfl_sync(0xffffffffu, h.SW, k);
                if (k == n - 1) SR = lane < k ? SWk : 1.0;
                else if (k > 0) SR = lane < k ? SR * SWk : SR;
            }
        }
        if (lane < n) {
            WalkDim w;
            // a node is kept iff its product is at least cutoff / R, taken
            // low enough that no rounding of the rest of the chain can lift a
            // dropped one to the cutoff; cutoff 0 keeps every node
            // (cut32 is within 2^-23 of the cutoff where it is not tiny: tiny
            // ones prune nothing; wide_bits, not a conversion: that would take
            // the FP64 pipe)
            const float thr = __fmul_rd(__fdiv_rd(cut32, R), 0.999999f);
            w.cp = cut32 > 1e-30f ? wide_bits(thr) : cut32 > 0.0f ? 0ll : LLONG_MIN;
            w.SR = SR;
            w.tw = h.tw;
            w.off = off;
            w.cb = h.ta * D.dim[lane].stride;
            w.stride = D.dim[lane].stride;
            w.magic = h.tw > 1 ? (uint32_t)((0x100000000ull + (unsigned)h.tw - 1) / (unsigned)h.tw) : 0u;
            w.pad = 0;
            S.h[lane] = w;
        }
        S.su = reinterpret_cast<double *>(S.ul + tsum);
        const int cs = (wl + 2) & ~1;
        S.pu = S.su + cs;
        S.pl = S.pu + cs;
        S.sf = S.pl + cs;
        S.su32 = reinterpret_cast<float *>(S.sf + cs);
        S.lists = reinterpret_cast<unsigned char *>(S.su + (sorted ? 5 * cs : 0));
        if (!empty) {
            for (int k = 0; k < n; ++k) {
                const unsigned long long p = __shfl_sync(0xffffffffu, (unsigned long long)it, k);
                const int twk = __shfl_sync(0xffffffffu, h.tw, k);
                const int fk = __shfl_sync(0xffffffffu, h.first, k);
                const int ok = __shfl_sync(0xffffffffu, off, k);
                const double2 *src = item_table(reinterpret_cast<unsigned char *>(p)) + fk;
                for (int e = lane; e < twk; e += 32) S.ul[ok + e] = src[e];
            }
            if (sorted) {
                unsigned char *pl = reinterpret_cast<unsigned char *>(
                    __shfl_sync(0xffffffffu, (unsigned long long)it, n - 1));
                const int tl = __shfl_sync(0xffffffffu, h.tw, n - 1);
                const double *src = item_sorted(pl, wl);
                for (int e = lane; e <= tl; e += 32) {
                    const double x = e < tl ? src[e] : 0.0;
                    S.su[e] = x;
                    S.su32[e] = lead32(x);
                    S.pu[e] = src[e + 2 * (wl + 1)];
                    S.pl[e] = src[e + 3 * (wl + 1)];
                    S.sf[e] = src[e + 4 * (wl + 1)];
                }
            }
        }
        __syncwarp();
        if (EMIT) {
            const int64_t base = A.row_ptr[row], len = A.row_ptr[row + 1] - base;
            if (base < 0 || len < 0 || (A.capacity >= 0 && base + len > A.capacity)) {
                if (lane == 0) atomicOr(A.status, IMPACT_STATUS_EMIT_MISMATCH);
            } else {
                const Out64 out{A.col + base, A.lo + base, A.up + base, len};
                Sums64 none;
                int64_t written = 0;
                bool ok = true;
                if (!empty) ok = walk_row64<true>(S, n, lane, none, out, written, keep, false);
                if (lane == 0 && (!ok || written != len))
                    atomicOr(A.status, ok ? IMPACT_STATUS_EMIT_MISMATCH : IMPACT_STATUS_INTERNAL);
            }
        } else {
            Sums64 acc;
            const Out64 none{nullptr, nullptr, nullptr, 0};
            int64_t w0 = 0;
            bool ok = true;
            if (!empty) ok = walk_row64<false>(S, n, lane, acc, none, w0, keep, sorted);
            const int cnt = __reduce_add_sync(0xffffffffu, acc.cnt);
            double sum[3] = {acc.drop, acc.sup, acc.slo};
            warp_sums(sum, lane);
            if (lane == 0) A.row_ptr[row] = ok ? cnt : 0;
            if (lane < 3) A.acc[lane * A.rows + row] = sum[0];
            if (lane == 0 && !ok) atomicOr(A.status, IMPACT_STATUS_INTERNAL);
        }
        __syncwarp();   // every lane is done with the row's tables
    }
}

int blocks_for(const void *kernel, int threads, size_t smem, int64_t items, int per_block)
{
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem);
    const int64_t want = (items + per_block - 1) / per_block;
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * std::max(occ, 1)));
}

}  // namespace

namespace impact {

int64_t size_items64(ImpactDesc &D)
{
    const int n = D.n;
    int64_t bytes = 0, tsum = 0;
    for (int d = 0; d < n; ++d) {
        ImpactDim &g = D.dim[d];
        const bool sorted = d == n - 1 && is_sorted_dim(D.cutoff32, g.w64);
        g.group = g.w64 + 1 <= 8 ? 8 : g.w64 + 1 <= 16 ? 16 : 32;
        tsum += g.w64;
        const int64_t st = kItemHead + 16 * (int64_t)g.w64 + (sorted ? 40 * (int64_t)(g.w64 + 1) : 0);
        g.item_stride = (int)std::min<int64_t>((st + 15) / 16 * 16, INT32_MAX / 2 / 16 * 16);
        g.item_off = bytes;
        bytes = g.n_items > kItemsMax / g.item_stride || bytes > kItemsMax
                    ? kItemsMax + 1 : bytes + g.n_items * (int64_t)g.item_stride;
    }
    // a window box too wide for a warp's shared memory, or tables beyond a fixed
    // size (images that are nearly all distinct, on large grids), keep the
    // per-pair evaluation, which needs no scratch
    D.walk64 = tsum <= kTablesMax && walk64_bytes(D) <= kSmemWarp && bytes <= kItemsMax;
    return D.walk64 ? bytes : 0;
}

int64_t walk64_bytes(const ImpactDesc &D)
{
    int64_t tsum = 0;
    for (int d = 0; d < D.n; ++d) tsum += D.dim[d].w64;
    const int wl = D.dim[D.n - 1].w64;
    return (warp_bytes64(D.n, tsum, wl, is_sorted_dim(D.cutoff32, wl)) + 15) / 16 * 16;
}

cudaError_t launch_items64(const BatchIndex *d_index, int64_t units, uint32_t *status,
                           cudaStream_t stream)
{
    if (units <= 0) return cudaSuccess;
    const int g = blocks_for((const void *)items_fp64, 256, 0, units, 8);
    items_fp64<<<g, 256, 0, stream>>>(d_index, status);
    return cudaGetLastError();
}

cudaError_t launch_terms64(const BatchIndex *d_index, int64_t rows, const double *acc,
                           const RowOutputs &o, const ScanHead &scan, cudaStream_t stream)
{
    if (rows <= 0) return cudaSuccess;
    const int g = blocks_for((const void *)terms_fp64, kTermThreads, 0, rows, kTermThreads);
    terms_fp64<<<scan.tiles + g, kTermThreads, 0, stream>>>(
        d_index, acc, o.sink_lo, o.sink_up, o.trunc, o.flags, o.status, scan);
    return cudaGetLastError();
}

cudaError_t launch_walk64(const BatchIndex *d_index, int64_t row_begin, int64_t row_end,
                          int warp_smem, bool emit, const RowOutputs &o, double *acc,
                          int64_t rows, unsigned long long *counter, cudaStream_t stream)
{
    const int64_t span = row_end - row_begin;
    if (span <= 0) return cudaSuccess;
    const int warps = std::max(1, std::min(kWarps, 200 * 1024 / std::max(warp_smem, 1)));
    const size_t smem = (size_t)warp_smem * warps;
    const void *k = emit ? (const void *)walk_fp64<true> : (const void *)walk_fp64<false>;
    cudaError_t e = allow_smem(k);
    if (e != cudaSuccess) return e;
    Walk64Args A;
    A.B = d_index;
    A.warp_smem = warp_smem;
    A.row_ptr = o.row_ptr;
    A.col = o.col;
    A.lo = (double *)o.lo;
    A.up = (double *)o.up;
    A.acc = acc;
    A.rows = rows;
    A.status = o.status;
    A.capacity = o.capacity;
    A.total_at = o.total_at;
    A.row_begin = row_begin;
    A.row_end = row_end;
    A.next_row = counter;
    const int g = blocks_for(k, warps * 32, smem, span, warps);
    A.row_block = (int)std::max<int64_t>(1, std::min<int64_t>(4, span / ((int64_t)g * warps * 64)));
    if (emit) walk_fp64<true><<<g, warps * 32, smem, stream>>>(A);
    else walk_fp64<false><<<g, warps * 32, smem, stream>>>(A);
    return cudaGetLastError();
}

}  // namespace impact
