// mc_keys.cuh -- exact decisions of the sampled-noise kernels: the cell of a
// coordinate, and the least draw that moves an image end past an edge, as
// integer keys that order like the doubles.
#pragma once
#include <math.h>
#include <stdint.h>

namespace mckeys {

// Order-preserving integer key of a finite double (-0 and +0 share key 0):
// x < y exactly when key(x) < key(y). Comparisons of keys are integer work,
// which matters here: FP64 issue is scarce on this part.
__device__ __forceinline__ long long dkey(double x)
{
    if (x == 0.0) return 0;
    const long long b = __double_as_longlong(x);
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffll);
}

// Cell of a coordinate: -1 below the domain, N above it, else the i with
// E_i <= y < E_{i+1} (the last cell also holds y == E_N). A first guess from
// the nominal width, corrected against the edges themselves.
__device__ __forceinline__ int cell_of(const double *__restrict__ E, int N, double inv_h, double y)
{
    if (y < E[0]) return -1;
    if (y > E[N]) return N;
    int i = (int)fmin(fmax(floor((y - E[0]) * inv_h), 0.0), (double)(N - 1));
    while (i > 0 && y < E[i]) --i;
    while (i < N - 1 && y >= E[i + 1]) ++i;
    return i;
}

// Neighbouring doubles of a finite x (bit arithmetic; 0 steps to the least
// subnormal of either sign).
__device__ __forceinline__ double step_up(double x)
{
    if (x == 0.0) return __longlong_as_double(1ll);
    const long long b = __double_as_longlong(x);
    return __longlong_as_double(x > 0.0 ? b + 1 : b - 1);
}
__device__ __forceinline__ double step_down(double x)
{
    if (x == 0.0) return -__longlong_as_double(1ll);
    const long long b = __double_as_longlong(x);
    return __longlong_as_double(x > 0.0 ? b - 1 : b + 1);
}

// The least double w whose rounded sum w + m reaches the edge E (gt: passes
// it). RN addition is monotone in w, so these w form an up-set; the guess
// E - m is moved a few ulps, and bisection over the keys' order finishes the
// rare case where the guess is far off (|m| much larger than |E - m|).
__device__ __forceinline__ double threshold_of(double m, double E, bool gt)
{
    auto ok = [&](double w) {
        const double y = w + m;
        return gt ? y > E : y >= E;
    };
    double w = E - m;
    for (int k = 0; k < 2; ++k) {
        if (ok(w)) {
            const double p = step_down(w);
            if (!ok(p)) return w;
            w = p;
        } else {
            w = step_up(w);
        }
    }
    // bracket [lo, hi] with ok(hi) and not ok(lo), then bisection on the
    // order of doubles (the sign is handled by the keys' order)
    double span = fmax(fabs(m), fabs(E)) * 0x1p-50 + 0x1p-1000;
    double lo = w - span, hi = w + span;
    for (int k = 0; k < 64 && ok(lo); ++k) lo -= (span *= 2.0);
    for (int k = 0; k < 64 && !ok(hi); ++k) hi += (span *= 2.0);
    for (int k = 0; k < 128; ++k) {
        const long long kl = dkey(lo), kh = dkey(hi);
        if (kh - kl <= 1) break;
        // midpoint in key order, back to a double
        const long long km = kl + (kh - kl) / 2;
        const double mid = km >= 0 ? __longlong_as_double(km)
                                   : __longlong_as_double(km ^ 0x7fffffffffffffffll);
        if (ok(mid)) hi = mid; else lo = mid;
    }
    return hi;
}

}  // namespace mckeys
