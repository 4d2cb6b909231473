// The 32 x 32 diagonal block of a Cholesky panel (schur.cu), factorised in shared memory by the warps of one block.  Plain
// C++ between the barriers: tests/test_chol_panel_races.py compiles it for the host and checks the accesses.
#pragma once

namespace wpccc {

// v -= l conj(u): one step of the Cholesky factor's element (i, j) with l = L[i][k], u = L[j][k]
static __device__ __forceinline__ float2 chol_step(float2 v, float2 l, float2 u) {
    v.x -= l.x * u.x + l.y * u.y;
    v.y -= l.y * u.x - l.x * u.y;
    return v;
}
static __device__ __forceinline__ double2 chol_step(double2 v, double2 l, double2 u) {
    v.x = fma(-l.x, u.x, fma(-l.y, u.y, v.x));
    v.y = fma(-l.y, u.x, fma(l.x, u.y, v.y));
    return v;
}

// (sqrt(d), 1 / sqrt(d)); in FP64 by two Newton-Raphson steps r <- r + r (1 - d r^2) / 2 from the FP32 reciprocal square
// root: an FP64 square root and division are long serial chains on this part's FP64 pipe.  The square root is d r, within
// two units in the last place, not the correctly rounded one.
static __device__ __forceinline__ float2 sqrt_and_inverse(float d) {
    const float s = sqrt(d);
    return make_float2(s, 1.f / s);
}
static __device__ __forceinline__ double2 sqrt_and_inverse(double d) {
    double r;
    if (d > 1e-30 && d < 1e30) {
        r = (double)rsqrtf((float)d);
        r = fma(0.5 * r, fma(-d * r, r, 1.0), r);
        r = fma(0.5 * r, fma(-d * r, r, 1.0), r);
    } else {
        r = rsqrt(d);
    }
    return make_double2(d * r, r);
}

// sL[col * ld + row], lower triangle of nb <= 32 rows: the block <- its factor; s_inv[k] <- 1 / L[k][k]; the first
// non-positive pivot (taken as 1) to *s_info, counted from k0 + 1.  By all threads of a block of WARPS warps, row = lane:
// column k is scaled by the first warp, the columns j > k belong to the warps in turn (an FP64 instruction holds a
// quarter's pipe for 64 cycles per warp, so the steps are spread over all four).  Ends with a block barrier.
template <int WARPS, typename C2, typename R>
static __device__ __forceinline__ void chol_diag_block(C2* sL, int ld, R* s_inv, int* s_info, int k0, int nb, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    for (int k = 0; k < nb; ++k) {
        if (warp == 0) {
            R d = sL[k * ld + k].x;
            if (!(d > R(0))) {
                if (lane == 0 && *s_info == 0) *s_info = k0 + k + 1;
                d = R(1);
            }
            const C2 r = sqrt_and_inverse(d);
            __syncwarp();   // every lane has read the pivot before lane k stores its root there
            if (lane == k) {
                sL[k * ld + k] = C2{r.x, R(0)};
                s_inv[k] = r.y;
            } else if (lane > k && lane < nb) {
                const C2 l = sL[k * ld + lane];
                sL[k * ld + lane] = C2{l.x * r.y, l.y * r.y};
            }
        }
        __syncthreads();
        const C2 l = sL[k * ld + (lane < nb ? lane : 0)];
        for (int j = k + 1 + warp; j < nb; j += WARPS)
            if (lane >= j && lane < nb) sL[j * ld + lane] = chol_step(sL[j * ld + lane], l, sL[k * ld + j]);
        __syncthreads();
    }
}

}  // namespace wpccc
