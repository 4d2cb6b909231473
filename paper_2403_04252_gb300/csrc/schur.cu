// Schur-complement factorisation of the two-centre overlap matrix (solve mode WPCCC_SOLVE_SCHUR).
//
// S = [[I, K], [K^+, I]] (Eq. 1) is a Gram matrix, Hermitian positive definite.  Eliminating the target
// block gives the Schur complement C = I - K^+ K (N_P x N_P, Hermitian positive definite), factorised
// by Cholesky, C = L L^+.  Then S k = t is
//   k_P = C^{-1} (t_P - K^+ t_T),   k_T = t_T - K k_P,
// i.e. two matrix-vector products with K and two triangular solves with L per RK4 stage, instead of the
// pivoted LU of the whole S.  Per position: the rank-N_T update K^+ K of the lower triangle (4 N_P^2 N_T
// real flops) and the Cholesky ((4/3) N_P^3), against (8/3) N^3 for the LU of S.
//
// One cluster of thread blocks per system; L overwrites the lower triangle of S's projectile-projectile block
// (the identity block, which the propagation never reads otherwise); K stays in place.  The mixed-
// precision forms take the same factorisation in FP32 into a separate buffer, as the preconditioner of
// their FP64 iterative refinement.
#include <algorithm>

#include "chol_panel.cuh"
#include "cluster.cuh"
#include "wpccc_internal.cuh"

namespace wpccc {

constexpr int SC_NB = 32;          // Cholesky panel width
static_assert(SC_NB == 32, "the diagonal block is factorised with a row per lane");
constexpr int SC_THREADS = 256;
constexpr int SC_T = 64;           // update tile, complex elements; a thread holds 4 x 4 of them
constexpr int SC_LD = SC_T + 1;    // its stride in shared memory (no bank conflicts on either index)

template <typename R> struct SchurC;
template <> struct SchurC<double> { using type = double2; };
template <> struct SchurC<float> { using type = float2; };

template <typename R>
constexpr size_t schur_smem() {
    return sizeof(typename SchurC<R>::type) * (2 * SC_NB * SC_LD + SC_NB * (SC_NB + 1));
}

// C[m x m] -= sum_kk A(i, kk) B(kk, j) over the lower triangle (i >= j) of C, for a reduction of kd terms taken SC_NB at a
// time; the tiles that touch the triangle go to the cluster's blocks in turn.  Every element is one chain of
// multiply-adds over kk, then one subtraction, whatever block forms it.  A and B are element loaders; KFAST: memory
// runs along kk (else along the row or column).
template <typename R, bool KFAST, typename LA, typename LB>
__device__ void cta_update_lower(typename SchurC<R>::type* __restrict__ C, int ldc, int m, int kd, LA loadA, LB loadB,
                                 typename SchurC<R>::type* sA, typename SchurC<R>::type* sB) {
    using C2 = typename SchurC<R>::type;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, wrow = (tid >> 5) * 8;   // a warp holds eight rows
    const int rank = cluster_rank(), size = cluster_size();
    int t = 0;
    for (int i0 = 0; i0 < m; i0 += SC_T) {
        for (int j0 = 0; j0 <= i0; j0 += SC_T, ++t) {
            if (t % size != rank) continue;
            C2 acc[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[a][c] = C2{R(0), R(0)};
            for (int k0 = 0; k0 < kd; k0 += SC_NB) {
#pragma unroll 4
                for (int idx = tid; idx < SC_T * SC_NB; idx += SC_THREADS) {
                    const int ii = KFAST ? idx / SC_NB : idx % SC_T, kk = KFAST ? idx % SC_NB : idx / SC_T;
                    sA[kk * SC_LD + ii] = (i0 + ii < m && k0 + kk < kd) ? loadA(i0 + ii, k0 + kk) : C2{R(0), R(0)};
                    sB[kk * SC_LD + ii] = (j0 + ii < m && k0 + kk < kd) ? loadB(k0 + kk, j0 + ii) : C2{R(0), R(0)};
                }
                __syncthreads();
                // column groups of the warp that touch the triangle (all but above the diagonal of a diagonal tile); none
                // for rows past the end
                const int kn = i0 + wrow < m ? min(SC_NB, kd - k0) : 0;
                const int cn = i0 == j0 ? (wrow + 7) / 16 + 1 : 4;
#pragma unroll 2
                for (int kk = 0; kk < kn; ++kk) {
                    C2 av[4], bv[4];
#pragma unroll
                    for (int a = 0; a < 4; ++a) av[a] = sA[kk * SC_LD + ty * 4 + a];
#pragma unroll
                    for (int c = 0; c < 4; ++c) bv[c] = sB[kk * SC_LD + tx + 16 * c];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (c >= cn) break;
#pragma unroll
                        for (int a = 0; a < 4; ++a) {
                            acc[a][c].x = fma(av[a].x, bv[c].x, acc[a][c].x);
                            acc[a][c].x = fma(-av[a].y, bv[c].y, acc[a][c].x);
                            acc[a][c].y = fma(av[a].x, bv[c].y, acc[a][c].y);
                            acc[a][c].y = fma(av[a].y, bv[c].x, acc[a][c].y);
                        }
                    }
                }
                __syncthreads();
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const int i = i0 + ty * 4 + a;
                if (i >= m) continue;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int j = j0 + tx + 16 * c;
                    if (j >= m || j > i) continue;
                    C2* p = C + (size_t)i + (size_t)j * ldc;
                    C2 v = __ldcg(p);
                    v.x -= acc[a][c].x;
                    v.y -= acc[a][c].y;
                    *p = v;
                }
            }
        }
    }
}

// One system per cluster of blocks (cluster size 1 to 8).  R = double: D is S itself (FP64, in place).  R = float
// (preconditioner of the mixed-precision form): D is a separate FP32 N x N buffer that receives K rounded to FP32
// in its target-projectile block and the FP32 Cholesky factor in its projectile block; S is only read.
// given = true: D already holds K (in FP32, or in S) and the trailing matrix I - K^+ K in the projectile block's
// lower triangle (formed on the tensor cores); only the Cholesky factor is computed.
//
// Blocked right-looking Cholesky.  Per panel of 32 columns every block of the cluster factorises the 32 x 32
// diagonal block for itself (chol_panel.cuh: all warps, a row per lane, in shared memory), the rows below go to the blocks' threads, a
// row each (L21 = A21 L11^{-+}, column by column in registers or shared memory), and the trailing tiles to the
// blocks in turn: two cluster barriers per panel.  Every element goes through the same operations in the same order
// as an unblocked column-by-column elimination within the panel, for any cluster size.  The FP64 factor is left for the
// row-shared solves of the RK4 sweep: L below the diagonal blocks, L^+ above them, and in each 32 x 32 diagonal block
// the inverse of L's block (lower half) with its adjoint (upper half).
template <typename R>
__global__ void __launch_bounds__(SC_THREADS) k_schur_factor(int N, int N_T, const double2* Sall,
                                                             typename SchurC<R>::type* __restrict__ Dall,
                                                             int* __restrict__ info_all, bool given) {
    using C2 = typename SchurC<R>::type;
    extern __shared__ __align__(16) unsigned char sc_smem_raw[];
    C2* sA = reinterpret_cast<C2*>(sc_smem_raw);   // SC_NB * SC_LD
    C2* sB = sA + SC_NB * SC_LD;                   // SC_NB * SC_LD
    C2* sL = sB + SC_NB * SC_LD;                   // [col][row], stride SC_NB + 1: the panel's diagonal block
    __shared__ R s_inv[SC_NB];
    __shared__ int s_info;
    const int rank = cluster_rank(), size = cluster_size();
    const int sys = blockIdx.x / size, tid = threadIdx.x, lane = tid & 31;
    const int NP = N - N_T;
    const size_t mat = (size_t)N * N;
    C2* D = Dall + (size_t)sys * mat;
    C2* C = D + N_T + (size_t)N_T * N;           // projectile block, leading dimension N
    const C2* K = D + (size_t)N_T * N;           // K[i][j] = D[i][N_T + j], i < N_T
    if (tid == 0) s_info = 0;
    if (sizeof(R) == 4 && !given) {
        // K to FP32, identity into the lower triangle of the projectile block
        const double2* S = Sall + (size_t)sys * mat;
        for (size_t q = (size_t)rank * SC_THREADS + tid; q < (size_t)N_T * NP; q += (size_t)size * SC_THREADS) {
            const int i = (int)(q % N_T), j = (int)(q / N_T);
            const double2 a = S[(size_t)i + (size_t)(N_T + j) * N];
            D[(size_t)i + (size_t)(N_T + j) * N] = C2{(R)a.x, (R)a.y};
        }
        for (size_t q = (size_t)rank * SC_THREADS + tid; q < (size_t)NP * NP; q += (size_t)size * SC_THREADS) {
            const int i = (int)(q % NP), j = (int)(q / NP);
            if (i >= j) C[(size_t)i + (size_t)j * N] = C2{R(i == j ? 1 : 0), R(0)};
        }
        cluster_sync_all();
    }
    // C = I - K^+ K on the lower triangle (the block holds I already)
    if (!given)
        cta_update_lower<R, true>(
            C, N, NP, N_T,
            [&](int i, int kk) {   // (K^+)[i][kk] = conj(K[kk][i])
                const C2 a = __ldcg(K + (size_t)kk + (size_t)i * N);
                return C2{a.x, -a.y};
            },
            [&](int kk, int j) { return __ldcg(K + (size_t)kk + (size_t)j * N); }, sA, sB);
    cluster_sync_all();
    for (int k0 = 0; k0 < NP; k0 += SC_NB) {
        const int nb = min(SC_NB, NP - k0);
        for (int q = tid; q < SC_NB * SC_NB; q += SC_THREADS) {
            const int i = q & 31, j = q >> 5;
            if (j <= i && i < nb) sL[j * (SC_NB + 1) + i] = __ldcg(C + (size_t)(k0 + i) + (size_t)(k0 + j) * N);
        }
        __syncthreads();
        chol_diag_block<SC_THREADS / 32>(sL, SC_NB + 1, s_inv, &s_info, k0, nb, tid);
        // every block has read the diagonal block before one of them overwrites it with its factor
        cluster_sync_all();
        if (sizeof(R) == 4) {
            if (rank == 0)
                for (int q = tid; q < SC_NB * SC_NB; q += SC_THREADS) {
                    const int i = q & 31, j = q >> 5;
                    if (j <= i && i < nb) C[(size_t)(k0 + i) + (size_t)(k0 + j) * N] = sL[j * (SC_NB + 1) + i];
                }
        } else if (rank == (k0 / SC_NB) % size) {
            // FP64: the inverse of the diagonal block (lower half) and its adjoint (upper half).  A warp takes four
            // columns of the inverse, a row per lane.
            const int c0 = (tid >> 5) * 4;
            C2 x[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) x[c] = C2{R(lane == c0 + c ? 1 : 0), R(0)};
            for (int k = c0; k < nb; ++k) {
                const R inv = s_inv[k];
                const C2 l = lane > k && lane < nb ? sL[k * (SC_NB + 1) + lane] : C2{R(0), R(0)};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const R wr = __shfl_sync(0xffffffffu, x[c].x, k) * inv, wi = __shfl_sync(0xffffffffu, x[c].y, k) * inv;
                    if (lane == k) x[c] = C2{wr, wi};
                    x[c].x = fma(-l.x, wr, x[c].x);
                    x[c].x = fma(l.y, wi, x[c].x);
                    x[c].y = fma(-l.x, wi, x[c].y);
                    x[c].y = fma(-l.y, wr, x[c].y);
                }
            }
            if (lane < nb)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int j = c0 + c;
                    if (j > lane) continue;
                    C[(size_t)(k0 + lane) + (size_t)(k0 + j) * N] = x[c];
                    if (j < lane) C[(size_t)(k0 + j) + (size_t)(k0 + lane) * N] = C2{x[c].x, -x[c].y};
                }
        }
        // rows below (none when nb < SC_NB): 64 rows per pass through shared memory, [col][row]
        const int m2 = NP - (k0 + nb);
        for (int r0 = rank * SC_T; r0 < m2; r0 += size * SC_T) {
            C2* P = C + (size_t)(k0 + nb + r0) + (size_t)k0 * N;
            for (int idx = tid; idx < SC_T * SC_NB; idx += SC_THREADS) {
                const int ii = idx % SC_T, kk = idx / SC_T;
                if (r0 + ii < m2) sA[kk * SC_LD + ii] = __ldcg(P + ii + (size_t)kk * N);
            }
            __syncthreads();
            // column k scaled, then the columns j > k updated by four threads per row
            const int ii = tid & (SC_T - 1), part = tid >> 6;
            for (int k = 0; k < SC_NB; ++k) {
                const R inv = s_inv[k];
                C2 l = sA[k * SC_LD + ii];
                l = C2{l.x * inv, l.y * inv};
                for (int j = k + 1 + part; j < SC_NB; j += 4)
                    sA[j * SC_LD + ii] = chol_step(sA[j * SC_LD + ii], l, sL[k * (SC_NB + 1) + j]);
                __syncthreads();
                if (part == 0) sA[k * SC_LD + ii] = l;   // column k is not read again in this pass
            }
            __syncthreads();
            for (int idx = tid; idx < SC_T * SC_NB; idx += SC_THREADS) {
                const int iw = idx % SC_T, kk = idx / SC_T;
                if (r0 + iw < m2) P[iw + (size_t)kk * N] = sA[kk * SC_LD + iw];
            }
            if (sizeof(R) == 8)   // FP64: L^+ above the diagonal too, for the backward solves' row-wise reads
                for (int idx = tid; idx < SC_T * SC_NB; idx += SC_THREADS) {
                    const int kk = idx % SC_NB, iw = idx / SC_NB;
                    if (r0 + iw < m2) {
                        const C2 l = sA[kk * SC_LD + iw];
                        C[(size_t)(k0 + kk) + (size_t)(k0 + nb + r0 + iw) * N] = C2{l.x, -l.y};
                    }
                }
            __syncthreads();
        }
        if (m2 > 0) {
            cluster_sync_all();
            C2* C22 = C + (size_t)(k0 + nb) + (size_t)(k0 + nb) * N;
            const C2* L21 = C + (size_t)(k0 + nb) + (size_t)k0 * N;
            cta_update_lower<R, false>(
                C22, N, m2, nb, [&](int i, int kk) { return __ldcg(L21 + (size_t)i + (size_t)kk * N); },
                [&](int kk, int j) {
                    const C2 a = __ldcg(L21 + (size_t)j + (size_t)kk * N);
                    return C2{a.x, -a.y};
                },
                sA, sB);
            cluster_sync_all();
        }
    }
    if (tid == 0 && rank == 0) info_all[sys] = s_info;
}

// Blocks per system: doubled while there is about one block per SM or less, as long as each has a few 64 x 64 tiles.
// Factorisation in ms with 1, 2, 4 and 8 blocks (* the rule's), FP64 N_P = 190 with the update on the tensor cores:
//   20 systems 2.18 1.56* 1.27 1.88, 50 systems 2.31 1.68* 2.13 3.00, 120 systems 2.57 2.84* 4.12 5.78, 160 4.20* 4.26 5.10 7.78;
// FP32 N_P = 190: 50 systems 0.67 0.43* 0.36 0.53, 120 systems 0.69 0.49* 0.70 1.06, 160 0.78* 0.89 1.00 1.33;
// FP32 N_P = 811: 20 systems 13.0 7.8 5.2 4.1*, 50 systems 16.4 10.8 8.3* 9.0, 80 systems 19.7 14.2* 14.4 13.7;
// FP64 N_P = 811: 100 systems 120 113* 92 (four), 160 systems 218 168* 149, 180 systems 220* 171 153, 250 systems 228* 227 214.
static int schur_cluster(int NP, int batch, int sms) {
    const int tiles = ((NP + SC_T - 1) / SC_T) * ((NP + SC_T - 1) / SC_T + 1) / 2;
    int cl = 1;
    while (cl < 8 && cl * batch <= sms + sms / 16 && tiles >= 4 * cl) cl *= 2;
    return cl;
}

template <typename R>
static wpccc_status schur_launch(int N, int N_T, int batch, const double2* S, typename SchurC<R>::type* D, int* info,
                                 bool given, cudaStream_t st) {
    if (batch == 0) return WPCCC_OK;
    const int smem = (int)schur_smem<R>();
    if (smem > 48 * 1024)
        WPCCC_CUDA(cudaFuncSetAttribute(k_schur_factor<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    int device = 0, sms = 0;
    WPCCC_CUDA(cudaGetDevice(&device));
    WPCCC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    ClusterLaunch L(batch, schur_cluster(N - N_T, batch, sms), SC_THREADS, smem, st);
    WPCCC_CUDA(cudaLaunchKernelEx(&L.cfg, k_schur_factor<R>, N, N_T, S, D, info, given));
    return WPCCC_OK;
}

wpccc_status launch_schur_factor(int N, int N_T, int batch, double2* S, int* info, cudaStream_t st) {
    return schur_launch<double>(N, N_T, batch, S, S, info, false, st);
}

wpccc_status launch_schur_factor_f32(int N, int N_T, int batch, const double2* S, float2* D, int* info,
                                     cudaStream_t st) {
    return schur_launch<float>(N, N_T, batch, S, D, info, false, st);
}

wpccc_status launch_schur_cholesky(int N, int N_T, int batch, double2* S, int* info, cudaStream_t st) {
    return schur_launch<double>(N, N_T, batch, S, S, info, true, st);
}

wpccc_status launch_schur_cholesky_f32(int N, int N_T, int batch, float2* D, int* info, cudaStream_t st) {
    return schur_launch<float>(N, N_T, batch, nullptr, D, info, true, st);
}

}  // namespace wpccc
