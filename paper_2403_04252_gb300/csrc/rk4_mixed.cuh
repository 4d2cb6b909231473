// The stage operator of the refined Schur forms (RK_MIXED_SCHUR) on a cluster of one to eight blocks per path:
// k = -(i/v) x with S x = H y solved by FP64 iterative refinement preconditioned by the FP32 Schur factors
// (x_0 = 0, r = H y - S x_n, x_{n+1} = x_n + S_32^{-1} r).
//
// What bounds it: a stage reads H, S's off-diagonal blocks and, per sweep, the FP32 factors once (N = 1622: 90 MB), more
// than one SM can draw in flight, and the FP64 residual takes 8 N_T N_P FMAs at two per clock per SM.  So the rows of
// every product are shared out over the cluster; every vector is replicated in the blocks' shared memory and results
// are stored into all copies.  The FP32 preconditioner's operations are those of the one-block solve in the same
// order (per row or per warp), for any cluster size: two sweeps leave its rounding visible in the result.
// Measured, one block per path -> here, sweeps alone: p + H, N = 380, 32 paths of 16 steps 36 -> 22 ms (two blocks per
// path); C6+ + H, N = 1622, 16 paths of 4 steps 140 -> 43 ms (four).
#pragma once

#include "rk4_fp64.cuh"

namespace wpccc {

static __device__ __forceinline__ void rc_bcast_f(const RcCluster& cl, float2* p, float2 v) {
    if (cl.size == 1) {
        *p = v;
        return;
    }
    const uint32_t a = smem_u32(p);
    for (int r = 0; r < cl.size; ++r) {
        uint32_t q;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(q) : "r"(a), "r"(r));
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};\n" ::"r"(q), "f"(v.x), "f"(v.y) : "memory");
    }
}

// rc_matvec in double-float arithmetic (matvec_df's terms; each group's compensated sum, the groups added in FP64).
template <typename F>
static __device__ __forceinline__ void rc_matvec_df(const double2* __restrict__ M, size_t ld, int nr, int nc,
                                                    const float4* ys, double2* part, F epi) {
    if (nr <= 0) return;
    const int tid = threadIdx.x;
    const int rb = min(RC_THREADS / RC_G, (nr + 7) & ~7);
    const int slot = tid % rb, grp = tid / rb;
    for (int base = 0; base < nr; base += rb) {
        const int row = base + slot;
        if (grp < RC_G && row < nr) {
            f32x2 s = x2_pack(0.f, 0.f), c = x2_pack(0.f, 0.f);   // (re, im)
            const double2* p = M + row + (size_t)grp * ld;
            const size_t step = (size_t)RC_G * ld;
#pragma unroll 8
            for (int j = grp; j < nc; j += RC_G, p += step) {
                const double2 m = *p;
                const float2 mr = split_bits(m.x), mi = split_bits(m.y);
                const float4 q = ys[j];   // (Re y hi, Re y lo, Im y hi, Im y lo)
                dot2_acc_x2(s, c, x2_pack(mr.x, mr.x), x2_pack(mr.y, mr.y), x2_pack(q.x, q.z), x2_pack(q.y, q.w));
                dot2_acc_x2(s, c, x2_pack(-mi.x, mi.x), x2_pack(-mi.y, mi.y), x2_pack(q.z, q.x), x2_pack(q.w, q.y));
            }
            float sr, si, cr, ci;
            x2_unpack(s, sr, si);
            x2_unpack(c, cr, ci);
            part[tid] = make_double2((double)sr + (double)cr, (double)si + (double)ci);
        }
        __syncthreads();
        rc_reduce(part, rb, base, nr, epi);
        __syncthreads();
    }
}

// d <- S_32^{-1} d (replicated, N entries) from the FP32 Schur factors D (K, and L below the projectile block's diagonal).
// u, w: scratch of N - N_T (replicated); blk: 32 x 32.
static __device__ __noinline__ void rc_schur_solve_f32(const RcCluster& cl, const float2* __restrict__ D, int N, int N_T,
                                                       float2* d, float2* u, float2* w, float2* blk) {
    const int NP = N - N_T, np = (NP + 31) / 32, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int WARPS = RC_THREADS / 32;
    const float2* __restrict__ K = D + (size_t)N_T * N;
    const float2* __restrict__ L = K + N_T;
    // u_P = t_P - K^+ t_T, a warp per column of K
    for (int j = cl.rank * WARPS + warp; j < NP; j += cl.size * WARPS) {
        float re = 0, im = 0;
        const float2* col = K + (size_t)j * N;
#pragma unroll 8
        for (int i = lane; i < N_T; i += 32) {
            const float2 a = col[i], b = d[i];
            re = fma(a.x, b.x, re);
            re = fma(a.y, b.y, re);
            im = fma(a.x, b.y, im);
            im = fma(-a.y, b.x, im);
        }
        for (int o = 16; o > 0; o >>= 1) {
            re += __shfl_xor_sync(0xffffffffu, re, o);
            im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        if (lane == 0) {
            float2 q = d[N_T + j];
            q.x -= re;
            q.y -= im;
            rc_bcast_f(cl, u + j, q);
        }
    }
    cl.sync();
    auto diag = [&](int p, bool back) {
        const int kb = 32 * p, nb = min(32, NP - kb);
        for (int q = tid; q < 32 * 32; q += RC_THREADS) {
            const int i = q & 31, j = q >> 5;
            if (i < nb && j <= i) blk[q] = L[(size_t)(kb + i) + (size_t)(kb + j) * N];
        }
        __syncthreads();
        if (warp == 0) {
            const int ln = lane < nb ? lane : 0;
            float2 v = u[kb + ln];
            const float rd = 1.f / blk[ln * 32 + ln].x;
            if (!back) {
                for (int j = 0; j < nb; ++j) {
                    if (lane == j) {
                        v.x *= rd;
                        v.y *= rd;
                    }
                    const float vr = __shfl_sync(0xffffffffu, v.x, j);
                    const float vi = __shfl_sync(0xffffffffu, v.y, j);
                    if (lane > j && lane < nb) {
                        const float2 l = blk[j * 32 + lane];
                        v.x = fma(-l.x, vr, v.x);
                        v.x = fma(l.y, vi, v.x);
                        v.y = fma(-l.x, vi, v.y);
                        v.y = fma(-l.y, vr, v.y);
                    }
                }
            } else {
                for (int j = nb - 1; j >= 0; --j) {
                    if (lane == j) {
                        v.x *= rd;
                        v.y *= rd;
                    }
                    const float vr = __shfl_sync(0xffffffffu, v.x, j);
                    const float vi = __shfl_sync(0xffffffffu, v.y, j);
                    if (lane < j) {
                        const float2 l = blk[lane * 32 + j];   // L[j][lane], conjugated below
                        v.x = fma(-l.x, vr, v.x);
                        v.x = fma(-l.y, vi, v.x);
                        v.y = fma(-l.x, vi, v.y);
                        v.y = fma(l.y, vr, v.y);
                    }
                }
            }
            if (lane < nb) rc_bcast_f(cl, w + kb + lane, v);
        }
    };
    // L z = u: a thread per own row, the panel's row entries loaded before the barrier that makes z known
    for (int p = 0; p < np; ++p) {
        const int kb = 32 * p, nb = min(32, NP - kb);
        const int q0 = rc_first_after(p, cl.rank, cl.size), cnt = rc_count(q0, np, cl.size);
        if (p % cl.size == cl.rank) diag(p, false);
        auto row_of = [&](int s) { return (q0 + (s >> 5) * cl.size) * 32 + (s & 31); };
        float2 a[32];
        const int r0 = row_of(tid);
        const bool on = tid < cnt * 32 && r0 < NP;   // rows below the panel: nb = 32 whenever there are any
#pragma unroll
        for (int j = 0; j < 32; ++j) a[j] = on ? L[(size_t)r0 + (size_t)(kb + j) * N] : make_float2(0.f, 0.f);
        cl.sync();
        for (int s = tid; s < cnt * 32; s += RC_THREADS) {
            const int r = row_of(s);
            if (r >= NP) continue;
            float2 x = u[r];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const float2 l = s == tid ? a[j] : L[(size_t)r + (size_t)(kb + j) * N], b = w[kb + j];
                x.x = fma(-l.x, b.x, x.x);
                x.x = fma(l.y, b.y, x.x);
                x.y = fma(-l.x, b.y, x.y);
                x.y = fma(-l.y, b.x, x.y);
            }
            u[r] = x;
        }
        (void)nb;
        __syncthreads();
    }
    // L^+ x = z: a warp per own row above the panel, lanes over its 32 entries
    for (int r = tid; r < NP; r += RC_THREADS)
        if ((r >> 5) % cl.size == cl.rank) u[r] = w[r];
    __syncthreads();
    for (int p = np - 1; p >= 0; --p) {
        const int kb = 32 * p, nb = min(32, NP - kb), cnt = rc_count(cl.rank, p, cl.size);
        if (p % cl.size == cl.rank) diag(p, true);
        auto row_of = [&](int s) { return (cl.rank + (s >> 5) * cl.size) * 32 + (s & 31); };
        constexpr int PRE = 8;
        float2 a[PRE];
#pragma unroll
        for (int q = 0; q < PRE; ++q) {
            const int s = warp + q * WARPS;
            a[q] = s < cnt * 32 && lane < nb ? L[(size_t)(kb + lane) + (size_t)row_of(s) * N] : make_float2(0.f, 0.f);
        }
        cl.sync();
        const float2 b = lane < nb ? w[kb + lane] : make_float2(0.f, 0.f);
        auto row = [&](int s, float2 l) {
            float re = 0, im = 0;
            if (lane < nb) {
                re = l.x * b.x + l.y * b.y;
                im = l.x * b.y - l.y * b.x;
            }
            for (int o = 16; o > 0; o >>= 1) {
                re += __shfl_xor_sync(0xffffffffu, re, o);
                im += __shfl_xor_sync(0xffffffffu, im, o);
            }
            if (lane == 0) {
                float2 q = u[row_of(s)];
                q.x -= re;
                q.y -= im;
                u[row_of(s)] = q;
            }
        };
#pragma unroll
        for (int q = 0; q < PRE; ++q)
            if (warp + q * WARPS < cnt * 32) row(warp + q * WARPS, a[q]);
        for (int s = warp + PRE * WARPS; s < cnt * 32; s += WARPS)
            row(s, lane < nb ? L[(size_t)(kb + lane) + (size_t)row_of(s) * N] : make_float2(0.f, 0.f));
        __syncthreads();
    }
    // x_T = t_T - K x_P, a thread per row
    int lo, hi;
    cl.rows(N_T, lo, hi);
    for (int i = lo + tid; i < hi; i += RC_THREADS) {
        float re = 0, im = 0;
#pragma unroll 16
        for (int j = 0; j < NP; ++j) {
            const float2 a = K[(size_t)i + (size_t)j * N];
            const float2 b = w[j];
            re = fma(a.x, b.x, re);
            re = fma(-a.y, b.y, re);
            im = fma(a.x, b.y, im);
            im = fma(a.y, b.x, im);
        }
        float2 q = d[i];
        q.x -= re;
        q.y -= im;
        rc_bcast_f(cl, d + i, q);
    }
    for (int j = tid; j < NP; j += RC_THREADS) d[N_T + j] = w[j];
    cl.sync();
}

// x = S^{-1} H y (replicated): H y into b (in double-float arithmetic when df_rhs), then `iters` refinement sweeps; the
// last sweep's correction is checked against the solution (refine_check) when tol > 0.  Scratch, N entries each: b, r, d
// and u, w (N - N_T); blk: 1024 float2, used for partial sums too.
static __device__ __noinline__ void rc_schur_refined(const RcCluster& cl, const double2* __restrict__ S64,
                                                     const float2* __restrict__ D32, const double2* __restrict__ Hm, int N,
                                                     int N_T, int iters, const double2* y, double2* b, double2* x,
                                                     double2* r, float2* d, float2* u, float2* w, float2* blk,
                                                     double tol, int* flags, bool df_rhs) {
    const int tid = threadIdx.x;
    double2* part = reinterpret_cast<double2*>(blk);
    int lo, hi;
    cl.rows(N, lo, hi);
    if (df_rhs) {
        float4* ys = reinterpret_cast<float4*>(r);
        for (int j = tid; j < N; j += RC_THREADS) {
            const float2 p = split_bits(y[j].x), q = split_bits(y[j].y);
            ys[j] = make_float4(p.x, p.y, q.x, q.y);
        }
        __syncthreads();
        rc_matvec_df(Hm + lo, N, hi - lo, N, ys, part, [&](int i, double2 v) { cl.bcast(b + lo + i, v); });
    } else {
        rc_matvec(Hm + lo, N, hi - lo, N, y, part, [&](int i, double2 v) { cl.bcast(b + lo + i, v); });
    }
    cl.sync();
    for (int it = 0; it < iters; ++it) {
        const double2* rr = b;
        if (it > 0) {
            // r = b - S x: only the off-diagonal blocks of S are read
            cl.rows(N_T, lo, hi);
            rc_matvec(S64 + lo + (size_t)N_T * N, N, hi - lo, N - N_T, x + N_T, part, [&](int i, double2 v) {
                const int g = lo + i;
                cl.bcast(r + g, make_double2(b[g].x - x[g].x - v.x, b[g].y - x[g].y - v.y));
            });
            cl.rows(N - N_T, lo, hi);
            rc_matvec(S64 + N_T + lo, N, hi - lo, N_T, x, part, [&](int i, double2 v) {
                const int g = N_T + lo + i;
                cl.bcast(r + g, make_double2(b[g].x - x[g].x - v.x, b[g].y - x[g].y - v.y));
            });
            cl.sync();
            rr = r;
        }
        for (int i = tid; i < N; i += RC_THREADS) d[i] = make_float2((float)rr[i].x, (float)rr[i].y);
        __syncthreads();
        rc_schur_solve_f32(cl, D32, N, N_T, d, u, w, blk);
        double dm = 0.0, xm = 0.0;
        for (int i = tid; i < N; i += RC_THREADS) {
            const double2 dx = make_double2((double)d[i].x, (double)d[i].y);
            x[i] = it == 0 ? dx : make_double2(x[i].x + dx.x, x[i].y + dx.y);
            dm = fmax(dm, fmax(fabs(dx.x), fabs(dx.y)));
            xm = fmax(xm, fmax(fabs(x[i].x), fabs(x[i].y)));
        }
        __syncthreads();
        if (it > 0 && it == iters - 1 && tol > 0.0) refine_check(dm, xm, tol, cl.rank == 0 ? flags : nullptr);
    }
}

}  // namespace wpccc
