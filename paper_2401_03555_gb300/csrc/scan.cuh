// scan.cuh -- the row-pointer scan in pieces of one block: exclusive scan of the
// per-row counts, in place in row_ptr, by tiles of kScanTile rows.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.h"

namespace rowscan {

constexpr int kScanTile = 4096;

// Exclusive prefix of v over the block (T threads) and the block's total.
template <int T>
__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t *sh, int64_t &total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        int64_t s = lane < T / 32 ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        sh[lane] = s;
    }
    __syncthreads();
    int64_t before = (w > 0 ? sh[w - 1] : 0) + x - v;
    total = sh[T / 32 - 1];
    __syncthreads();
    return before;
}

// The sum of tile `tile` of v[n].
template <int T>
__device__ __forceinline__ void tile_sum(const int64_t *v, int64_t n, int64_t tile, int64_t *tsum)
{
    __shared__ int64_t sh[32];
    const int64_t base = tile * kScanTile;
    int64_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanTile / T; ++k) {
        const int64_t i = base + k * T + threadIdx.x;
        if (i < n) s += v[i];
    }
    int64_t total;
    block_excl_scan<T>(s, sh, total);
    if (threadIdx.x == 0) tsum[tile] = total;
}

// Row pointers of tile `tile` from its counts and the sum of those before it;
// the last tile also stores the total, in v[n] and *also.
template <int T>
__device__ __forceinline__ void tile_apply(int64_t *v, int64_t n, int64_t tile, int64_t before,
                                           bool last, int64_t *also)
{
    __shared__ int64_t sh[32];
    constexpr int E = kScanTile / T;
    const int64_t base = tile * kScanTile + (int64_t)threadIdx.x * E;
    int64_t loc[E];
    int64_t s = 0;
#pragma unroll
    for (int k = 0; k < E; ++k) {
        loc[k] = base + k < n ? v[base + k] : 0;
        s += loc[k];
    }
    int64_t sum;
    int64_t ex = block_excl_scan<T>(s, sh, sum) + before;
#pragma unroll
    for (int k = 0; k < E; ++k) {
        if (base + k < n) v[base + k] = ex;
        ex += loc[k];
    }
    if (last && threadIdx.x == 0) {
        v[n] = before + sum;
        if (also) *also = before + sum;
    }
}

// The scan's first pass as blocks of another kernel: block b < S.tiles sums tile
// b, or with one tile does the whole scan.
template <int T>
__device__ __forceinline__ void first_pass(const impact::ScanHead &S)
{
    if (S.tiles == 1) tile_apply<T>(S.row_ptr, S.n, 0, 0, true, S.also);
    else tile_sum<T>(S.row_ptr, S.n, blockIdx.x, S.tsum);
}

}  // namespace rowscan
