// Geometry helpers of the element kernels and of their adjoint (one definition, so both pick the
// same node radii and interpolation stencils).
#pragma once

#include <cuda_runtime.h>

namespace wpccc {

// ---------------------------------------------------------------------------
// geometry shared by the kernels; explicit round-to-nearest operations so that
// the interpolation stencils are chosen from exactly the same radii as a plain
// IEEE evaluation of the same formulas (no contraction into FMA)
// ---------------------------------------------------------------------------
static __device__ inline double dist_R(double b, double z) {
    return __dsqrt_rn(__dadd_rn(__dmul_rn(b, b), __dmul_rn(z, z)));
}

// Start of the 5-point stencil at x (two nodes left of the largest j with r[j] <= x) by one warp, in every lane; Lagrange
// weight a in lane a < 5.  x <= r[Nr - 1].
static __device__ inline void stencil5_warp(const double* __restrict__ r, int Nr, double x, int lane, int& s, double& L) {
    int lo = -1, hi = Nr;   // r[lo] <= x < r[hi]
    while (hi - lo > 1) {
        const int step = (hi - lo + 32) / 33, p = lo + (lane + 1) * step;
        const int c = __popc(__ballot_sync(0xffffffffu, p < hi && r[p] <= x));
        lo += c * step;
        hi = min(hi, lo + step);
    }
    s = min(max(lo - 2, 0), Nr - 5);
    const int a = min(lane, 4);
    double p = 1.0;
    for (int c = 0; c < 5; ++c)
        if (c != a) p *= (x - r[s + c]) / (r[s + a] - r[s + c]);
    L = p;
}

// The same stencil with the Lagrange denominators 1/prod_{c != a}(r_{s+a} - r_{s+c}) read from a
// table made at set-up (inv_den[s][a], 5 per stencil start), so no division per interpolation.
static __device__ inline bool stencil5_fast(const double* __restrict__ r, const double* __restrict__ inv_den, int Nr,
                                     double x, int& s, double L[5]) {
    if (x > r[Nr - 1]) return false;
    int lo = -1, hi = Nr;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        // numbers >= 0 compare like their bit patterns, which leaves the FP64 pipe free
        if (__double_as_longlong(r[mid]) <= __double_as_longlong(x)) lo = mid;
        else hi = mid;
    }
    s = min(max(lo - 2, 0), Nr - 5);
    double dx[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) dx[k] = x - r[s + k];
#pragma unroll
    for (int a = 0; a < 5; ++a) {
        double p = inv_den[(size_t)s * 5 + a];
#pragma unroll
        for (int c = 0; c < 5; ++c)
            if (c != a) p *= dx[c];
        L[a] = p;
    }
    return true;
}

}  // namespace wpccc
