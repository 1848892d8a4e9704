// mc_masks.cu -- sampled-noise rows by draw masks (impact_build_mc, Sec. 4.1).
//
// The cells a draw's moved box meets are a box of cells, so a draw counts for
// a target iff it does in every dimension: with one bit per draw, the count of
// target t is popc(AND_d up_d[t_d]) over the words of the draws, and the bits
// of a prefix of dimensions are shared by everything below it.
//
//   mc_items  per distinct image of a dimension (impact_desc.h) the window of
//             cells within reach and, for each of them, the draws whose moved
//             interval meets it (up) and lies in it (lo); the draws that stay
//             in the domain and that leave it whole; and how many cells each
//             draw meets. Decisions by the integer keys of the per-edge
//             thresholds, as in the per-row kernel.
//   mc_walk   one warp per row, one lane per word of 32 draws (up to four): the
//             window's cells as a prefix tree in C order, a node dropped as
//             soon as fewer than kmin draws are left. The dropped mass is the
//             draws' met cells in all, less those of the kept targets
//             (integers: exact). The count pass keeps each row's targets and
//             counts (8 bytes a pair) in a scratch whose size the host bounds;
//             the emit pass turns them into pairs, and walks again only the
//             rows that found no room.
//
// The per-row histogram (kernels.cu) pays per draw: 2n threshold searches and
// about 2^n shared-memory atomics. This pays per tree node one AND, one popc
// and one warp sum over all the draws at once. Room 7^5 (151k rows, 1024 draws,
// cutoff 2e-3): 84.4 -> 4.19 ms per call (items 0.11, count 3.4, emit 0.13; with
// both passes walking 5.9). The count is bound by popc and the warp sums, 16
// lanes a clock each.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "impact_desc.h"
#include "kernels.h"
#include "mc_keys.cuh"
#include "rowmath.cuh"

namespace {

using namespace rowmath;
using impact::McKeep;
using impact::McMasks;
using impact::RowOutputs;

// warps per block: the level masks of a block stay within 32 KB
__host__ __device__ constexpr int warps_of(int nw) { return nw >= 4 ? 4 : 8; }

// An item: {o, ext} in 16 bytes, then rows of W = 32 NW words: the draws inside,
// those that leave whole, up[cap], lo[cap]; then one byte per draw, the cells
// it meets. cap = min(cells, 64): wider windows are refused by the row.
struct McItem {
    int o, ext;
    int pad[2];
};

__device__ __forceinline__ uint32_t *item_words(unsigned char *it)
{
    return reinterpret_cast<uint32_t *>(it + sizeof(McItem));
}

__global__ void __launch_bounds__(128)
mc_items(const ImpactDesc *__restrict__ Dp, McMasks K, const long long *__restrict__ keys,
         int64_t S, const double *__restrict__ range, unsigned char *__restrict__ items)
{
    __shared__ long long thr_lo[IMPACT_MC_EDGES_MAX + 1], thr_hi[IMPACT_MC_EDGES_MAX + 1];
    const ImpactDesc &D = *Dp;
    const int lane = threadIdx.x & 31, W = 32 * K.nw;
    for (int64_t u = blockIdx.x; u < K.first[D.n]; u += gridDim.x) {
        int d = 0;
        while (u >= K.first[d + 1]) ++d;
        const ImpactDim &g = D.dim[d];
        const double *E = D.edges + g.edge_off;
        const int64_t c = u - K.first[d];
        int idx[IMPACT_MAX_DIM], j = 0;
        decode_item(D, d, c, idx, j);
        double lo, hi;
        image_dim<false>(D, c, idx, j, d, lo, hi);
        const double mlo = fmin(lo, hi), mhi = fmax(lo, hi);   // ordered ends
        const int a = max(mckeys::cell_of(E, g.N, g.inv_h, range[2 * d] + mlo), 0);
        const int b = min(mckeys::cell_of(E, g.N, g.inv_h, range[2 * d + 1] + mhi), g.N - 1);
        const int ext = b >= a ? b - a + 1 : 0;
        unsigned char *it = items + K.off[d] + c * K.stride[d];
        if (threadIdx.x == 0) *reinterpret_cast<McItem *>(it) = McItem{a, ext, {0, 0}};
        if (ext == 0 || ext > IMPACT_MC_EDGES_MAX) continue;   // the same for the whole block
        for (int k = threadIdx.x; k < 2 * (ext + 1); k += blockDim.x) {
            const int e = k >> 1, end = k & 1, edge = a + e;
            const long long t = mckeys::dkey(
                mckeys::threshold_of(end ? mhi : mlo, E[edge], edge == g.N));
            if (end) thr_hi[e] = t; else thr_lo[e] = t;
        }
        __syncthreads();
        uint32_t *w0 = item_words(it);
        unsigned char *met = reinterpret_cast<unsigned char *>(w0 + (2 + 2 * K.cap[d]) * W);
        for (int w = threadIdx.x >> 5; w < W; w += blockDim.x >> 5) {
            const int64_t s = (int64_t)w * 32 + lane;
            const bool valid = s < S;
            const long long key = valid ? keys[(int64_t)d * S + s] : 0;
            // beyond edge k at the image's low / high end
            bool lo_k = valid && key >= thr_lo[0], hi_k = valid && key >= thr_hi[0];
            const bool below = a == 0 && !hi_k;            // whole image left of the domain
            bool in = valid && (a > 0 || lo_k);
            int n_met = 0;
            for (int t = 0; t < ext; ++t) {
                const bool lo_n = valid && key >= thr_lo[t + 1], hi_n = valid && key >= thr_hi[t + 1];
                const bool up = hi_k && !lo_n, inside = lo_k && !hi_n;
                n_met += up;
                const unsigned mu = __ballot_sync(0xffffffffu, up);
                const unsigned ml = __ballot_sync(0xffffffffu, inside);
                if (lane == 0) {
                    w0[(2 + t) * W + w] = mu;
                    w0[(2 + K.cap[d] + t) * W + w] = ml;
                }
                lo_k = lo_n;
                hi_k = hi_n;
            }
            const bool top = a + ext == g.N;
            in = in && !(top && hi_k);
            const bool out = valid && (below || (top && lo_k));
            const unsigned mi = __ballot_sync(0xffffffffu, in);
            const unsigned mo = __ballot_sync(0xffffffffu, out);
            if (lane == 0) {
                w0[w] = mi;
                w0[W + w] = mo;
            }
            met[s] = (unsigned char)n_met;
        }
        __syncthreads();   // the thresholds are rewritten for the next item
    }
}

// Scratch of the count pass: entries {column, u | l << 16}, claimed in chunks by
// the warps; seg[row] is the row's first entry (-1: not kept).
constexpr int kChunk = 2048;

template <bool EMIT, int NW>
__global__ void __launch_bounds__(32 * warps_of(NW))
mc_walk(const ImpactDesc *__restrict__ Dp, int64_t rows, McMasks K,
        unsigned char *__restrict__ items, int64_t S, const double *__restrict__ val,
        const float *__restrict__ val_dn, const float *__restrict__ val_up, unsigned kmin,
        int hist_cap, McKeep keep_in, RowOutputs o)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int W = 32 * NW;
    // per warp and level: the draws left (up and lo)
    __shared__ uint32_t level[warps_of(NW)][IMPACT_MAX_DIM][2][W];
    const ImpactDesc &D = *Dp;
    const int n = D.n, lane = threadIdx.x & 31;
    auto &L = level[threadIdx.x >> 5];
    if (EMIT && o.capacity >= 0 && o.row_ptr[o.total_at] > o.capacity) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(o.status, IMPACT_STATUS_CAPACITY);
        return;
    }
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const double dS = (double)S;
    int64_t chunk_at = 0, chunk_end = 0;   // this warp's scratch
    for (int64_t row = warp0; row < rows; row += nwarps) {
        if (EMIT) {
            const int64_t seg = keep_in.seg[row];
            if (seg >= 0) {   // kept by the count pass
                const int64_t base = o.row_ptr[row], len = o.row_ptr[row + 1] - base;
                for (int64_t i = lane; i < len; i += 32) {
                    const uint2 e = keep_in.entries[seg + i];
                    const unsigned u = e.y & 0xffffu, l = e.y >> 16;
                    o.col[base + i] = (int32_t)e.x;
                    if (D.prec == PREC_FP64_PLAIN) {
                        ((double *)o.up)[base + i] = val[u];
                        ((double *)o.lo)[base + i] = val[l];
                    } else {
                        ((float *)o.up)[base + i] = val_up[u];
                        ((float *)o.lo)[base + i] = val_dn[l];
                    }
                }
                continue;
            }
        }
        // lane d: the item of dimension d
        McItem h{0, 1, {0, 0}};
        unsigned char *it = nullptr;
        int stride = 0;
        {
            int idx[IMPACT_MAX_DIM], j;
            decode_row(D, row, idx, j);
            if (lane < n) {
                it = items + K.off[lane] + item_of(D, row, idx, j, lane) * K.stride[lane];
                h = *reinterpret_cast<const McItem *>(it);
                stride = D.dim[lane].stride;
            }
        }
        int64_t H = 1;
        for (int d = 0; d < n; ++d) H *= __shfl_sync(kAll, h.ext, d);   // at most the grid's cells
        const bool wide = __any_sync(kAll, h.ext > IMPACT_MC_EDGES_MAX);
        if (H > hist_cap || wide) {   // window too large: counted as empty, the call fails
            if (lane == 0) {
                atomicOr(o.status, IMPACT_STATUS_MC_WINDOW);
                if (!EMIT) {
                    o.row_ptr[row] = 0;
                    keep_in.seg[row] = 0;
                }
            }
            continue;
        }
        if (H == 0) {   // every draw leaves the domain whole
            if (!EMIT && lane == 0) {
                o.row_ptr[row] = 0;
                keep_in.seg[row] = 0;
                o.sink_lo[row] = o.sink_up[row] = dS / dS;
                o.trunc[row] = 0.0;
                if (o.flags) o.flags[row] = 0u;
            }
            continue;
        }
        auto words = [&](int d) {
            return item_words(reinterpret_cast<unsigned char *>(
                __shfl_sync(kAll, (unsigned long long)it, d)));
        };
        // the draws that stay in the domain, that leave it whole, and the
        // cells all draws meet
        unsigned inside = 0, outside = 0, met = 0;
        bool store = false;
        if (!EMIT) {
            uint32_t in[NW], out[NW];
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                in[i] = kAll;
                out[i] = 0;
            }
            for (int d = 0; d < n; ++d) {
                const uint32_t *wd = words(d);
#pragma unroll
                for (int i = 0; i < NW; ++i) {
                    in[i] &= wd[lane + 32 * i];
                    out[i] |= wd[W + lane + 32 * i];
                }
            }
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                inside += __popc(in[i]);
                outside += __popc(out[i]);
            }
            for (int q = 0; q < 8 * NW; ++q) {   // four draws per word
                unsigned p0 = 1, p1 = 1, p2 = 1, p3 = 1;
                for (int d = 0; d < n; ++d) {
                    const uint32_t v = words(d)[(2 + 2 * K.cap[d]) * W + q * 32 + lane];
                    p0 *= v & 0xffu;
                    p1 *= (v >> 8) & 0xffu;
                    p2 *= (v >> 16) & 0xffu;
                    p3 *= v >> 24;
                }
                met += p0 + p1 + p2 + p3;
            }
            inside = __reduce_add_sync(kAll, inside);
            outside = __reduce_add_sync(kAll, outside);
            met = __reduce_add_sync(kAll, met);
            // room for the row's targets: no more than the window has cells,
            // and each takes kmin of the met cells
            const int64_t most = min(H, (int64_t)(met / kmin));
            if (chunk_at + most > chunk_end) {
                unsigned long long at_ = 0;
                const int64_t take = max(most, (int64_t)kChunk);
                if (lane == 0) at_ = atomicAdd(keep_in.used, (unsigned long long)take);
                chunk_at = (int64_t)__shfl_sync(kAll, at_, 0);
                chunk_end = chunk_at + take;
                if (chunk_end > keep_in.cap) chunk_at = chunk_end = 0;   // no room left
            }
            store = chunk_at + most <= chunk_end;
        }
        // counts of `m` cells whose masks start at wd under the draws X: lane t
        // gets cell t's (two cells share a warp sum: a count fits 16 bits)
        auto counts = [&](const uint32_t *wd, int m, const uint32_t (&X)[NW]) {
            unsigned u = 0;
#pragma unroll 2
            for (int t = 0; t < m; t += 2) {
                unsigned c0 = 0, c1 = 0;
#pragma unroll
                for (int i = 0; i < NW; ++i) {
                    c0 += __popc(X[i] & wd[t * W + lane + 32 * i]);
                    if (t + 1 < m) c1 += __popc(X[i] & wd[(t + 1) * W + lane + 32 * i]);
                }
                const unsigned both = __reduce_add_sync(kAll, c0 | (c1 << 16));
                if ((lane >> 1) == (t >> 1)) u = both;
            }
            return lane & 1 ? u >> 16 : u & 0xffffu;
        };
        unsigned kept = 0, kept_sum = 0;
        int64_t at = EMIT ? o.row_ptr[row] : chunk_at;
        const int64_t end = EMIT ? o.row_ptr[row + 1] : 0;
        // the last dimension: every cell of its window under a node's draws
        const uint32_t *const wl = words(n - 1);
        const int ext_l = __shfl_sync(kAll, h.ext, n - 1), off_l = __shfl_sync(kAll, h.o, n - 1);
        const int st_l = __shfl_sync(kAll, stride, n - 1);
        auto leaf = [&](const uint32_t (&M)[NW], const uint32_t (&ML)[NW], int col0) {
            for (int t0 = 0; t0 < ext_l; t0 += 32) {
                const int m = min(32, ext_l - t0);
                const unsigned u = counts(wl + (2 + t0) * W, m, M);
                const bool keep = lane < m && u >= kmin;
                if (!EMIT) {
                    if (keep) {
                        ++kept;
                        kept_sum += u;
                    }
                    if (!store) continue;
                }
                const unsigned bal = __ballot_sync(kAll, keep);
                if (bal == 0) continue;
                const unsigned l = counts(wl + (2 + K.cap[n - 1] + t0) * W, m, ML);
                const int64_t p = at + __popc(bal & ((1u << lane) - 1u));
                if (!EMIT) {
                    if (keep)
                        keep_in.entries[p] = make_uint2(
                            (unsigned)(col0 + (off_l + t0 + lane) * st_l), u | (l << 16));
                } else if (keep && p < end) {
                    o.col[p] = col0 + (off_l + t0 + lane) * st_l;
                    if (D.prec == PREC_FP64_PLAIN) {
                        ((double *)o.up)[p] = val[u];
                        ((double *)o.lo)[p] = val[l];
                    } else {
                        ((float *)o.up)[p] = val_up[u];
                        ((float *)o.lo)[p] = val_dn[l];
                    }
                }
                at += __popc(bal);
            }
        };
        // lane k: the cells of level k with enough draws left and not walked
        // yet (bits from its window's first cell), the column of its node
        unsigned my_a0 = 0, my_a1 = 0;
        int my_col = 0, k = 0;
        auto open = [&](int d, const uint32_t (&M)[NW]) {
            const uint32_t *wd = words(d);
            const int ext = __shfl_sync(kAll, h.ext, d);
            const int m0 = min(32, ext), m1 = ext - m0;
            const unsigned u0 = counts(wd + 2 * W, m0, M);
            const unsigned a0 = __ballot_sync(kAll, lane < m0 && u0 >= kmin);
            unsigned a1 = 0;
            if (m1 > 0) {
                const unsigned u1 = counts(wd + 34 * W, m1, M);
                a1 = __ballot_sync(kAll, lane < m1 && u1 >= kmin);
            }
            if (lane == d) {
                my_a0 = a0;
                my_a1 = a1;
            }
        };
        uint32_t M[NW], ML[NW];
#pragma unroll
        for (int i = 0; i < NW; ++i) M[i] = ML[i] = kAll;
        if (n == 1) leaf(M, ML, 0);
        else open(0, M);
        while (n > 1) {
            const unsigned a0 = __shfl_sync(kAll, my_a0, k), a1 = __shfl_sync(kAll, my_a1, k);
            if ((a0 | a1) == 0) {
                if (k == 0) break;
                --k;
                continue;
            }
            const int t = a0 ? __ffs(a0) - 1 : 31 + __ffs(a1);
            if (lane == k) {
                if (a0) my_a0 = a0 & (a0 - 1);
                else my_a1 = a1 & (a1 - 1);
            }
            const uint32_t *wd = words(k) + (2 + t) * W + lane;
            const int col = (k > 0 ? __shfl_sync(kAll, my_col, k - 1) : 0) +
                            (__shfl_sync(kAll, h.o, k) + t) * __shfl_sync(kAll, stride, k);
#pragma unroll
            for (int i = 0; i < NW; ++i) {   // a lane reads back its own words only
                M[i] = (k > 0 ? L[k - 1][0][lane + 32 * i] : kAll) & wd[32 * i];
                if (EMIT || store)
                    ML[i] = (k > 0 ? L[k - 1][1][lane + 32 * i] : kAll) & wd[K.cap[k] * W + 32 * i];
            }
            if (k == n - 2) {
                leaf(M, ML, col);
                continue;
            }
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                L[k][0][lane + 32 * i] = M[i];
                if (EMIT || store) L[k][1][lane + 32 * i] = ML[i];
            }
            if (lane == k) my_col = col;
            ++k;
            open(k, M);
        }
        if (EMIT) {
            if (lane == 0 && at != end) atomicOr(o.status, IMPACT_STATUS_EMIT_MISMATCH);
            continue;
        }
        kept = __reduce_add_sync(kAll, kept);
        kept_sum = __reduce_add_sync(kAll, kept_sum);
        if (lane == 0) {
            keep_in.seg[row] = store ? chunk_at : -1;
            o.row_ptr[row] = kept;
            o.sink_lo[row] = (double)outside / dS;
            o.sink_up[row] = (double)((unsigned)S - inside) / dS;
            o.trunc[row] = (double)(met - kept_sum) / dS;
            if (o.flags) o.flags[row] = 0u;
        }
        if (store) chunk_at += kept;   // kept is the whole row's in every lane
    }
}

template <bool EMIT, int NW>
cudaError_t launch(const ImpactDesc *d_desc, int64_t rows, const McMasks &K, unsigned char *items,
                   int64_t S, const double *val, const float *val_dn, const float *val_up,
                   unsigned kmin, const McKeep &keep, const RowOutputs &o, cudaStream_t stream)
{
    constexpr int kWarps = warps_of(NW), kThreads = 32 * kWarps;
    const void *k = (const void *)mc_walk<EMIT, NW>;
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kThreads, 0);
    const int64_t g = std::min<int64_t>((rows + kWarps - 1) / kWarps, (int64_t)sms * std::max(occ, 1));
    mc_walk<EMIT, NW><<<(unsigned)g, kThreads, 0, stream>>>(d_desc, rows, K, items, S, val, val_dn,
                                                            val_up, kmin, IMPACT_MC_HIST_MAX, keep, o);
    return cudaGetLastError();
}

}  // namespace

namespace impact {

// The masks pay per tree node, so: a cutoff (kmin >= 1 prunes the tree), rows
// that share images, up to 4096 draws (four words per lane) and masks that stay
// near the L2 (256 MB at most). Else bytes stays 0. Room 6^5, 100 / 1000 / 4096
// draws, masks against histograms: cutoff 1e-6 (every met cell kept) 1.8 / 2.1 /
// 5.0 against 13.3 / 38.6 / 232 ms, cutoff 2e-2 1.7 / 1.6 / 3.4 against 13.1 /
// 38.6 / 232.
McMasks mc_masks(const ImpactDesc &D, int64_t S, double cutoff)
{
    McMasks K{};
    int64_t items = 0;
    K.nw = S <= 1024 ? 1 : S <= 2048 ? 2 : 4;
    for (int d = 0; d < D.n; ++d) {
        const ImpactDim &g = D.dim[d];
        K.cap[d] = std::min(g.N, IMPACT_MC_EDGES_MAX);
        K.stride[d] = (int)sizeof(McItem) + (2 + 2 * K.cap[d]) * 128 * K.nw + 1024 * K.nw;
        K.first[d + 1] = K.first[d] + g.n_items;
        K.off[d] = K.bytes;
        K.bytes += g.n_items * K.stride[d];
        items += g.n_items;
    }
    if (!(cutoff > 0.0) || S > 4096 || D.kind == KIND_IMAGES || items * 3 > D.rows * D.n ||
        K.bytes > ((int64_t)256 << 20))
        K.bytes = 0;
    return K;
}

// Entries the count pass may keep: 512 a row, 1 GB at most.
int64_t mc_keep_entries(int64_t rows)
{
    return std::min<int64_t>(std::max<int64_t>(rows * 512, 1 << 20), (int64_t)1 << 27);
}

cudaError_t launch_mc_items(const ImpactDesc *d_desc, int n, const McMasks &K,
                            const long long *keys, int64_t S, const double *range,
                            unsigned char *items, cudaStream_t stream)
{
    const int64_t g = std::min<int64_t>(K.first[n], 152 * 16);
    mc_items<<<(unsigned)g, 128, 0, stream>>>(d_desc, K, keys, S, range, items);
    return cudaGetLastError();
}

cudaError_t launch_mc_walk(const ImpactDesc *d_desc, bool emit, int64_t rows, const McMasks &K,
                           unsigned char *items, int64_t S, const double *val,
                           const float *val_dn, const float *val_up, unsigned kmin,
                           const McKeep &keep, const RowOutputs &o, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    if (K.nw == 1)
        return emit ? launch<true, 1>(d_desc, rows, K, items, S, val, val_dn, val_up, kmin, keep, o, st)
                    : launch<false, 1>(d_desc, rows, K, items, S, val, val_dn, val_up, kmin, keep, o, st);
    if (K.nw == 2)
        return emit ? launch<true, 2>(d_desc, rows, K, items, S, val, val_dn, val_up, kmin, keep, o, st)
                    : launch<false, 2>(d_desc, rows, K, items, S, val, val_dn, val_up, kmin, keep, o, st);
    return emit ? launch<true, 4>(d_desc, rows, K, items, S, val, val_dn, val_up, kmin, keep, o, st)
                : launch<false, 4>(d_desc, rows, K, items, S, val, val_dn, val_up, kmin, keep, o, st);
}

}  // namespace impact
