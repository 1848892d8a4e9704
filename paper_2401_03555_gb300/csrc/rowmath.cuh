// rowmath.cuh -- device arithmetic shared by the kernels that evaluate a
// build's definition in FP64: row and item numbering, the interval image of a
// source cell (Def. 3.1's box relaxation), the window of target cells and the
// Gaussian mass of a cell.
#pragma once
#include <math.h>
#include <stdint.h>

#include "impact_desc.h"

namespace rowmath {

__device__ __forceinline__ uint32_t fastdiv(uint32_t x, uint32_t m, int s)
{
    return (__umulhi(x, m) + x) >> s;   // exact for x < 2^31 (host-built m, s)
}

// Cell digits (C order) of a row, and the input index.
__device__ __forceinline__ void decode_row(const ImpactDesc &D, int64_t row, int *idx, int &j)
{
    uint32_t c;
    if (row < ((int64_t)1 << 31)) {
        c = fastdiv((uint32_t)row, D.inp_div_m, D.inp_div_s);
        j = (int)((uint32_t)row - c * (uint32_t)D.n_inputs);
    } else {
        const int64_t cell = row / D.n_inputs;
        j = (int)(row - cell * D.n_inputs);
        c = (uint32_t)cell;
    }
#pragma unroll
    for (int d = IMPACT_MAX_DIM - 1; d >= 0; --d) {
        if (d < D.n) {
            const uint32_t q = fastdiv(c, D.dim[d].div_m, D.dim[d].div_s);
            idx[d] = (int)(c - q * (uint32_t)D.dim[d].N);
            c = q;
        } else {
            idx[d] = 0;
        }
    }
}

// Item of dimension d that the row with these digits shares.
__device__ __forceinline__ int64_t item_of(const ImpactDesc &D, int64_t row, const int *idx, int j,
                                           int d)
{
    if (D.kind == KIND_IMAGES) return row;
    const ImpactDim &g = D.dim[d];
    int64_t c = D.cls[d * D.n_inputs + j];
#pragma unroll
    for (int k = 0; k < IMPACT_MAX_DIM; ++k)
        if (k < D.n) c += (int64_t)idx[k] * g.item_mul[k];
    return c;
}

// Digits and input of a row of item c (0 in the dimensions the image does not
// read: their terms are zeros in every cell, so the image is bitwise that of
// every row of the item).
__device__ __forceinline__ void decode_item(const ImpactDesc &D, int d, int64_t c, int *idx, int &j)
{
    const ImpactDim &g = D.dim[d];
    j = D.cls_rep[d * D.n_inputs + (int)(c % g.n_classes)];
    c /= g.n_classes;
#pragma unroll
    for (int k = IMPACT_MAX_DIM - 1; k >= 0; --k) {
        idx[k] = 0;
        if (k < D.n && g.item_mul[k] != 0) {
            idx[k] = (int)(c % D.dim[k].N);
            c /= D.dim[k].N;
        }
    }
}

// Interval image of f(., u_j) over the cell in dimension d.
//   SOUND: outward-rounded bounds of the exact image.
//   plain: round-to-nearest in the same operation order as the definition
//          (sum over k of the per-term range, then the input offset).
template <bool SOUND>
__device__ __forceinline__ void image_dim(const ImpactDesc &D, int64_t row, const int *idx, int j,
                                          int d, double &mlo, double &mhi)
{
    const int n = D.n;
    if (D.kind == KIND_AFFINE) {
        const int NM = D.n_max;
        if (SOUND) {
            double slo = 0.0, shi = 0.0;
            for (int k = 0; k < n; ++k) {
                int t = (d * n + k) * NM + idx[k];
                slo = __dadd_rd(slo, D.term_dn[t]);
                shi = __dadd_ru(shi, D.term_up[t]);
            }
            mlo = __dadd_rd(slo, D.off_dn[j * n + d]);
            mhi = __dadd_ru(shi, D.off_up[j * n + d]);
        } else {
            double slo = 0.0, shi = 0.0;
            for (int k = 0; k < n; ++k) {
                int t = ((d * n + k) * NM + idx[k]) * 2;
                slo = __dadd_rn(slo, D.term_rn[t]);
                shi = __dadd_rn(shi, D.term_rn[t + 1]);
            }
            mlo = __dadd_rn(slo, D.off_rn[j * n + d]);
            mhi = __dadd_rn(shi, D.off_rn[j * n + d]);
        }
    } else if (D.kind == KIND_UNICYCLE) {
        const double *E = D.edges + D.dim[d].edge_off;
        double xlo = E[idx[d]], xhi = E[idx[d] + 1];
        if (d == 2) {
            double om = D.inputs[j * D.m + 1];
            if (SOUND) { mlo = __dadd_rd(xlo, om); mhi = __dadd_ru(xhi, om); }
            else { mlo = __dadd_rn(xlo, om); mhi = __dadd_rn(xhi, om); }
        } else {
            const double *u = (SOUND ? D.uni_sd : D.uni_rn) + ((int64_t)idx[2] * D.n_inputs + j) * 4;
            double vlo = u[d * 2 + 0], vhi = u[d * 2 + 1];
            if (SOUND) { mlo = __dadd_rd(xlo, vlo); mhi = __dadd_ru(xhi, vhi); }
            else { mlo = __dadd_rn(xlo, vlo); mhi = __dadd_rn(xhi, vhi); }
        }
    } else {
        const double *im = D.images + (row * n + d) * 2;
        mlo = im[0];
        mhi = im[1];
    }
}

// Conservative window [a, b] of target cells in dimension d: any target whose
// cell lies entirely more than delta beyond the image has every upper factor
// below cutoff/2. One extra cell of slack on each side absorbs rounding.
__device__ __forceinline__ void window_dim(const ImpactDim &g, double mlo, double mhi, int &a,
                                           int &b)
{
    if (!(g.delta < INFINITY)) {
        a = 0;
        b = g.N - 1;
        return;
    }
    double xa = floor((mlo - g.delta - g.lo) * g.inv_h) - 1.0;
    double xb = floor((mhi + g.delta - g.lo) * g.inv_h) + 1.0;
    xa = fmin(fmax(xa, 0.0), (double)(g.N - 1));
    xb = fmin(fmax(xb, 0.0), (double)(g.N - 1));
    a = (int)xa;
    b = (int)xb;
    if (b < a) b = a - 1;   // empty
}

// Mass of a cell from its edges' arguments a <= b (in erf units around the
// mean) and fa = erfc(|a|), fb = erfc(|b|): the form whose terms are the small
// tails. Neighbouring cells share an edge, so one erfc per edge serves both.
__device__ __forceinline__ double mass64(double a, double fa, double b, double fb)
{
    if (a >= 0.0) return 0.5 * (fa - fb);
    if (b <= 0.0) return 0.5 * (fb - fa);
    return 1.0 - 0.5 * fa - 0.5 * fb;
}

// g(c, e; m) = Phi((e-m)/sigma) - Phi((c-m)/sigma), inv_s = 1/(sigma sqrt 2).
__device__ __forceinline__ double g64(double c, double e, double m, double inv_s)
{
    const double a = (c - m) * inv_s;
    const double b = (e - m) * inv_s;
    return mass64(a, erfc(fabs(a)), b, erfc(fabs(b)));
}

__device__ __forceinline__ double clampd(double x, double lo, double hi)
{
    return x < lo ? lo : (x > hi ? hi : x);
}

// Problem of a batch that owns global row x: begin[q] <= x < begin[q + 1].
__device__ __forceinline__ int find_problem(const int64_t *__restrict__ begin, int count,
                                            int64_t x)
{
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (begin[mid] <= x) lo = mid; else hi = mid - 1;
    }
    return lo;
}

}  // namespace rowmath
