// Batched complex linear solve S X = H with partial pivoting (the paper's ZGESV
// step of Eq. 4) in FP64, and the FP32 factorisation of the mixed-precision forms.
//
// Blocked right-looking elimination of the augmented matrix [S | H]:
//   for each panel of NB columns
//     1. unblocked LU of the panel with partial pivoting (largest |re|+|im|,
//        lowest row on ties, as LAPACK's izamax)
//     2. the panel's row interchanges applied to every other column of S and H
//     3. U12 = L11^{-1} A12 for the trailing columns of S and all columns of H
//     4. trailing update A22 -= L21 U12 (complex GEMM on the FP64 pipe)
//   then blocked back substitution X = U^{-1} Y on H.
// S is left holding L and U of P S = L U (LAPACK layout), H holds X.
//
// A system belongs to a cluster of one to eight blocks: the first factorises the panels, and the 32-column blocks of
// S and of H belong to the blocks in turn (interchanges, U12 and the trailing update of a column block need the panel
// only), so each panel takes two cluster barriers and the back substitution none.  One block per system leaves most
// of the chip idle for a small batch: at two FP64 multiply-adds per clock an SM needs 70 ms for one N = 380 system
// with N right-hand sides.  Every element goes through the same operations in the same order for any cluster size.
#include <algorithm>

#include "cluster.cuh"
#include "wpccc_internal.cuh"

namespace wpccc {

constexpr int NB = 32;            // panel width (the triangular solves map one row per lane)
static_assert(NB == 32, "NB must equal the warp size");
constexpr int LU_THREADS = 256;
constexpr int TM = 64, TN = 32;   // update tile, complex elements

template <typename R> struct LuC;
template <> struct LuC<double> { using type = double2; };
template <> struct LuC<float> { using type = float2; };

// C[m x n] -= A[m x k] * B[k x n], column-major, k <= NB, n <= TN, whole block cooperating.
template <typename C2>
__device__ void cta_gemm_sub(C2* __restrict__ C, int ldc, const C2* __restrict__ A, int lda, const C2* __restrict__ B,
                             int ldb, int m, int n, int k, C2* sA, C2* sB) {
    using R = decltype(C2().x);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const C2 zero = C2{R(0), R(0)};
    for (int idx = tid; idx < NB * TN; idx += LU_THREADS) {
        const int kk = idx % NB, jj = idx / NB;
        sB[kk * TN + jj] = (jj < n && kk < k) ? B[(size_t)kk + (size_t)jj * ldb] : zero;
    }
    for (int i0 = 0; i0 < m; i0 += TM) {
        for (int idx = tid; idx < TM * NB; idx += LU_THREADS) {
            const int ii = idx % TM, kk = idx / TM;
            sA[kk * TM + ii] = (i0 + ii < m && kk < k) ? __ldcg(A + (size_t)(i0 + ii) + (size_t)kk * lda) : zero;
        }
        __syncthreads();
        C2 acc[4][2];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 2; ++c) acc[a][c] = zero;
        for (int kk = 0; kk < k; ++kk) {
            C2 av[4], bv[2];
#pragma unroll
            for (int a = 0; a < 4; ++a) av[a] = sA[kk * TM + ty + 16 * a];
#pragma unroll
            for (int c = 0; c < 2; ++c) bv[c] = sB[kk * TN + tx + 16 * c];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    acc[a][c].x = fma(av[a].x, bv[c].x, acc[a][c].x);
                    acc[a][c].x = fma(-av[a].y, bv[c].y, acc[a][c].x);
                    acc[a][c].y = fma(av[a].x, bv[c].y, acc[a][c].y);
                    acc[a][c].y = fma(av[a].y, bv[c].x, acc[a][c].y);
                }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = i0 + ty + 16 * a;
            if (i >= m) continue;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int j = tx + 16 * c;
                if (j >= n) continue;
                C2* p = C + (size_t)i + (size_t)j * ldc;
                C2 v = *p;
                v.x -= acc[a][c].x;
                v.y -= acc[a][c].y;
                *p = v;
            }
        }
        __syncthreads();
    }
}

template <typename C2>
__device__ inline C2 crecip(C2 a) {
    const auto d = a.x * a.x + a.y * a.y;
    return C2{a.x / d, -a.y / d};
}
template <typename C2>
__device__ inline C2 cprod(C2 a, C2 b) {
    return C2{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
// x - l u
template <typename C2>
__device__ __forceinline__ C2 csub_prod(C2 x, C2 l, C2 u) {
    x.x = fma(-l.x, u.x, x.x);
    x.x = fma(l.y, u.y, x.x);
    x.y = fma(-l.x, u.y, x.y);
    x.y = fma(-l.y, u.x, x.y);
    return x;
}

// Order of |re| + |im| as an integer: the bits of a number >= 0; -1 for NaN, which is never a pivot while there is another.
__device__ __forceinline__ long long pivot_key(double v) { return v == v ? __double_as_longlong(v) : -1; }
__device__ __forceinline__ long long pivot_key(float v) { return v == v ? (long long)__float_as_int(v) : -1; }

// Unblocked LU with partial pivoting of the panel's nb columns from k0 (rows k0..N-1), by one block; pivots (1-based)
// to ipiv, the first zero pivot to *info.  An FP64 instruction holds its quarter of the SM's pipe for 64 cycles per warp, so
// the search for the pivot compares integers, and two lanes of one warp form the pivot's reciprocal (a division is some 30
// instructions) while the other warps interchange the rows.  Against the division in every warp and FP64 comparisons:
// N = 109, 200 factorisations 2.9 -> 2.4 ms; N = 380 with N right-hand sides, 24 systems 24.8 -> 24.2 ms.
template <typename C2>
__device__ void panel_lu(C2* __restrict__ A, int N, int k0, int nb, int* __restrict__ ipiv, int* info) {
    using R = decltype(C2().x);
    __shared__ long long red_v[LU_THREADS / 32];
    __shared__ int red_i[LU_THREADS / 32];
    __shared__ R s_inv[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int kk = 0; kk < nb; ++kk) {
        const int k = k0 + kk;
        long long best = -1;
        int bi = N;
        for (int i = k + tid; i < N; i += LU_THREADS) {
            const C2 a = A[(size_t)i + (size_t)k * N];
            const long long v = pivot_key(fabs(a.x) + fabs(a.y));
            if (v > best) {
                best = v;
                bi = i;
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const long long ov = __shfl_down_sync(0xffffffffu, best, off);
            const int oi = __shfl_down_sync(0xffffffffu, bi, off);
            if (ov > best || (ov == best && oi < bi)) {
                best = ov;
                bi = oi;
            }
        }
        if (lane == 0) {
            red_v[warp] = best;
            red_i[warp] = bi;
        }
        __syncthreads();
        best = red_v[0];
        bi = red_i[0];
        for (int w = 1; w < LU_THREADS / 32; ++w)
            if (red_v[w] > best || (red_v[w] == best && red_i[w] < bi)) {
                best = red_v[w];
                bi = red_i[w];
            }
        const int p = bi < N ? bi : k;
        if (tid == 0) {
            ipiv[k] = p + 1;
            if (best == 0 && *info == 0) *info = k + 1;
        }
        // the first warp: the pivot's reciprocal and this column's interchange; the next: the other columns'
        if (tid < 2) {
            const C2 piv = A[(size_t)p + (size_t)k * N];
            const R d = piv.x * piv.x + piv.y * piv.y;
            s_inv[tid] = (tid == 0 ? piv.x : -piv.y) / d;
            __syncwarp(3u);
            if (tid == 0 && p != k) {
                A[(size_t)p + (size_t)k * N] = A[(size_t)k + (size_t)k * N];
                A[(size_t)k + (size_t)k * N] = piv;
            }
        } else if (p != k && warp == 1 && lane < nb && lane != kk) {
            const int c = k0 + lane;
            const C2 t = A[(size_t)k + (size_t)c * N];
            A[(size_t)k + (size_t)c * N] = A[(size_t)p + (size_t)c * N];
            A[(size_t)p + (size_t)c * N] = t;
        }
        __syncthreads();
        if (best != 0) {
            const C2 inv = C2{s_inv[0], s_inv[1]};
            for (int i = k + 1 + tid; i < N; i += LU_THREADS) {
                C2* q = A + (size_t)i + (size_t)k * N;
                *q = cprod(*q, inv);
            }
        }
        __syncthreads();
        const int ncol = nb - kk - 1, nrow = N - k - 1;
        for (int idx = tid; idx < ncol * nrow; idx += LU_THREADS) {
            const int i = k + 1 + idx % nrow, j = k + 1 + idx / nrow;
            C2* q = A + (size_t)i + (size_t)j * N;
            *q = csub_prod(*q, A[(size_t)i + (size_t)k * N], A[(size_t)k + (size_t)j * N]);
        }
        __syncthreads();
    }
}

// One system per cluster.  R = double: Sall is factorised in place and, with Hall, S X = H solved.  R = float (the mixed
// forms' preconditioner): S is read in FP64, rounded to FP32 into Fall and factorised there; Hall is null.
template <typename R>
__global__ void __launch_bounds__(LU_THREADS) k_lu(int N, const double2* Sall, typename LuC<R>::type* Fall,
                                                   typename LuC<R>::type* __restrict__ Hall, int* __restrict__ ipiv_all,
                                                   int* __restrict__ info_all) {
    using C2 = typename LuC<R>::type;
    extern __shared__ __align__(16) unsigned char lu_smem[];
    C2* sA = reinterpret_cast<C2*>(lu_smem);   // TM * NB
    C2* sB = sA + TM * NB;                     // NB * TN
    C2* sT = sB + NB * TN;                     // NB * NB triangular block
    C2* sD = sT + NB * NB;                     // NB reciprocals of U's diagonal
    __shared__ int s_piv[NB];
    const int rank = cluster_rank(), size = cluster_size();
    const int sys = blockIdx.x / size, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int WARPS = LU_THREADS / 32;
    const size_t mat = (size_t)N * N;
    const C2 zero = C2{R(0), R(0)};
    C2* A = Fall + (size_t)sys * mat;
    C2* Bm = Hall ? Hall + (size_t)sys * mat : nullptr;
    int* ipiv = ipiv_all + (size_t)sys * N;
    int* info = info_all + sys;
    if (sizeof(R) == 4) {
        const double2* S = Sall + (size_t)sys * mat;
        for (size_t q = (size_t)rank * LU_THREADS + tid; q < mat; q += (size_t)size * LU_THREADS)
            A[q] = C2{(R)S[q].x, (R)S[q].y};
    }
    if (rank == 0 && tid == 0) *info = 0;
    cluster_sync_all();
    const int nbA = (N + NB - 1) / NB, nbH = Bm ? nbA : 0;   // column blocks of S, then of H
    for (int k0 = 0; k0 < N; k0 += NB) {
        const int nb = min(NB, N - k0), kb = k0 / NB;
        // ---- 1. panel factorisation
        if (rank == 0) panel_lu(A, N, k0, nb, ipiv, info);
        cluster_sync_all();
        if (tid < nb) s_piv[tid] = __ldcg(ipiv + k0 + tid) - 1;
        // L11 (unit lower) into shared memory
        for (int idx = tid; idx < NB * NB; idx += LU_THREADS) {
            const int i = idx % NB, j = idx / NB;
            sT[idx] = (i < nb && j < nb) ? __ldcg(A + (size_t)(k0 + i) + (size_t)(k0 + j) * N) : zero;
        }
        __syncthreads();
        // ---- 2. interchanges on this block's columns outside the panel (a warp per column block, a column per lane)
        for (int t = warp; t * size + rank < nbA + nbH; t += WARPS) {
            const int cb = t * size + rank;
            const int c = (cb < nbA ? cb : cb - nbA) * NB + lane;
            if (cb == kb || c >= N) continue;
            C2* col = (cb < nbA ? A : Bm) + (size_t)c * N;
            for (int kk = 0; kk < nb; ++kk) {
                const int p = s_piv[kk], k = k0 + kk;
                if (p != k) {
                    const C2 q = col[k];
                    col[k] = col[p];
                    col[p] = q;
                }
            }
        }
        __syncthreads();
        // ---- 3. U12 = L11^{-1} A12 for this block's trailing S columns and H columns: a warp per column, lane i holds
        //         row k0 + i; 4. their trailing update
        const int m = N - k0 - nb;
        for (int cb = rank; cb < nbA + nbH; cb += size) {
            if (cb <= kb) continue;
            C2* base = (cb < nbA ? A : Bm) + (size_t)(cb < nbA ? cb : cb - nbA) * NB * N;
            const int n = min(NB, N - (cb < nbA ? cb : cb - nbA) * NB);
            for (int c = warp; c < n; c += WARPS) {
                C2* col = base + (size_t)c * N + k0;
                C2 x = lane < nb ? col[lane] : zero;
                for (int j = 0; j < nb - 1; ++j) {
                    const C2 u = C2{__shfl_sync(0xffffffffu, x.x, j), __shfl_sync(0xffffffffu, x.y, j)};
                    if (lane > j) x = csub_prod(x, sT[j * NB + lane], u);
                }
                if (lane < nb) col[lane] = x;
            }
            __syncthreads();
            if (m > 0)
                cta_gemm_sub<C2>(base + k0 + nb, N, A + (size_t)(k0 + nb) + (size_t)k0 * N, N, base + k0, N, m, n, nb, sA, sB);
        }
        cluster_sync_all();
    }
    if (!Bm || __ldcg(info) != 0) return;   // factor only, or no solution for a singular system (as ZGESV)

    // ---- back substitution X = U^{-1} Y, every block on its own columns of H
    for (int kb = ((N - 1) / NB) * NB; kb >= 0; kb -= NB) {
        const int nb = min(NB, N - kb);
        for (int idx = tid; idx < NB * NB; idx += LU_THREADS) {
            const int i = idx % NB, j = idx / NB;
            sT[idx] = (i < nb && j < nb) ? __ldcg(A + (size_t)(kb + i) + (size_t)(kb + j) * N) : zero;
        }
        if (tid < NB) sD[tid] = tid < nb ? crecip(__ldcg(A + (size_t)(kb + tid) + (size_t)(kb + tid) * N)) : zero;
        __syncthreads();
        for (int cb = nbA + (rank + size - nbA % size) % size; cb < nbA + nbH; cb += size) {
            C2* base = Bm + (size_t)(cb - nbA) * NB * N;
            const int n = min(NB, N - (cb - nbA) * NB);
            for (int c = warp; c < n; c += WARPS) {
                C2* col = base + (size_t)c * N + kb;
                C2 x = lane < nb ? col[lane] : zero;
                for (int j = nb - 1; j >= 0; --j) {
                    if (lane == j) x = cprod(x, sD[j]);
                    const C2 u = C2{__shfl_sync(0xffffffffu, x.x, j), __shfl_sync(0xffffffffu, x.y, j)};
                    if (lane < j) x = csub_prod(x, sT[j * NB + lane], u);
                }
                if (lane < nb) col[lane] = x;
            }
            __syncthreads();
            if (kb > 0) cta_gemm_sub<C2>(base, N, A + (size_t)kb * N, N, base + kb, N, kb, n, nb, sA, sB);
        }
        __syncthreads();
    }
}

// Blocks per system: the size that finishes the batch soonest when a cluster's blocks sit on SMs of their own (the FP64
// pipe bounds the work, so blocks that share an SM gain nothing): ceil(batch / clusters the chip holds) / size, with at
// least two column blocks per block.  A cluster stays within a group of SMs, so the chip holds fewer clusters than SMs /
// size: 24 systems, N = 380, with N right-hand sides take 96, 50, 35, 27, 25, 34 and 34 ms with 1, 2, 3, 4, 5, 6 and 8
// (the rule takes 5; SMs / systems would be 6), 60 systems 98, 51, 65, 50, 62, 61 and 58 (2).
template <typename R>
static int lu_cluster(int N, int batch, bool rhs, int (&held)[9], cudaStream_t st) {
    if (held[1] == 0) {
        for (int size = 1; size <= 8; ++size) {
            ClusterLaunch L(1, size, LU_THREADS, 120 * 1024, st);   // more than half an SM's shared memory
            if (cudaOccupancyMaxActiveClusters(&held[size], k_lu<R>, &L.cfg) != cudaSuccess) {
                cudaGetLastError();
                held[size] = 0;
            }
        }
    }
    const int blocks = (N + NB - 1) / NB * (rhs ? 2 : 1);
    int best = 1;
    double t = 0.0;
    for (int size = 1; size <= std::max(1, std::min(8, blocks / 2)); ++size) {
        if (held[size] < 1) continue;
        const double s = (double)((batch + held[size] - 1) / held[size]) / size;
        if (size == 1 || s < 0.95 * t) {
            t = s;
            best = size;
        }
    }
    return best;
}

template <typename R>
static wpccc_status lu_launch(int N, int batch, const double2* S, typename LuC<R>::type* F, typename LuC<R>::type* H,
                              int* ipiv, int* info, cudaStream_t st) {
    using C2 = typename LuC<R>::type;
    if (batch == 0) return WPCCC_OK;
    const int smem = (int)(sizeof(C2) * (TM * NB + NB * TN + NB * NB + NB));
    WPCCC_CUDA(cudaFuncSetAttribute(k_lu<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, std::max(smem, 120 * 1024)));
    // clusters an empty chip holds, by size, of the device that this thread last used
    static thread_local int held[9] = {}, device = -1;
    int now = 0;
    WPCCC_CUDA(cudaGetDevice(&now));
    if (now != device) {
        held[1] = 0;
        device = now;
    }
    ClusterLaunch L(batch, lu_cluster<R>(N, batch, H != nullptr, held, st), LU_THREADS, smem, st);
    WPCCC_CUDA(cudaLaunchKernelEx(&L.cfg, k_lu<R>, N, S, F, H, ipiv, info));
    return WPCCC_OK;
}

// The 32 x 32 diagonal blocks of P S = L U replaced by the inverses of their triangles: strictly below the diagonal the
// unit lower block's inverse (its unit diagonal implied), from the diagonal on the upper block's.  One block per (panel,
// system), a warp per four columns of an inverse, a row per lane.  The RK4 sweep applies them instead of solving with the
// triangles.  As issued (both triangles, all lanes) the complex multiply-adds are 5200 / N^2 of the factorisation's: half of
// it at N = 109 (0.3 ms beside 2.4 for 200 systems: all panels at once), 4 % at N = 380.
__global__ void __launch_bounds__(256) k_lu_invert_diag(int N, double2* __restrict__ LU) {
    __shared__ double2 blk[NB][NB + 1];   // [column][row]
    const int k0 = blockIdx.x * NB, nb = min(NB, N - k0), lane = threadIdx.x & 31, c0 = (threadIdx.x >> 5) * 4;
    double2* A = LU + (size_t)blockIdx.y * N * N + (size_t)k0 + (size_t)k0 * N;
    for (int q = threadIdx.x; q < NB * NB; q += 256) {
        const int i = q & 31, j = q >> 5;
        blk[j][i] = i < nb && j < nb ? A[(size_t)i + (size_t)j * N] : make_double2(i == j ? 1.0 : 0.0, 0.0);
    }
    __syncthreads();
    const double2 inv = crecip(blk[lane][lane]);
    double2 l[4], u[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) l[c] = u[c] = make_double2(lane == c0 + c ? 1.0 : 0.0, 0.0);
    for (int k = c0; k < nb; ++k) {
        const double2 a = lane > k ? blk[k][lane] : make_double2(0.0, 0.0);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double2 w = make_double2(__shfl_sync(0xffffffffu, l[c].x, k), __shfl_sync(0xffffffffu, l[c].y, k));
            l[c] = csub_prod(l[c], a, w);
        }
    }
    for (int k = min(c0 + 3, nb - 1); k >= 0; --k) {
        const double2 a = lane < k ? blk[k][lane] : make_double2(0.0, 0.0);
        const double2 d = make_double2(__shfl_sync(0xffffffffu, inv.x, k), __shfl_sync(0xffffffffu, inv.y, k));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double2 w = cprod(make_double2(__shfl_sync(0xffffffffu, u[c].x, k), __shfl_sync(0xffffffffu, u[c].y, k)), d);
            if (lane == k) u[c] = w;
            u[c] = csub_prod(u[c], a, w);
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (lane < nb && c0 + c < nb) A[(size_t)lane + (size_t)(c0 + c) * N] = lane > c0 + c ? l[c] : u[c];
}

wpccc_status launch_lu_invert_diag(int N, int batch, double2* LU, cudaStream_t st) {
    if (batch == 0) return WPCCC_OK;
    k_lu_invert_diag<<<dim3((N + NB - 1) / NB, batch), 256, 0, st>>>(N, LU);
    WPCCC_CHECK_LAUNCH("k_lu_invert_diag");
    return WPCCC_OK;
}

wpccc_status launch_factor_f32(int N, int batch, const double2* S, float2* LU, int* ipiv, int* info, cudaStream_t st) {
    return lu_launch<float>(N, batch, S, LU, nullptr, ipiv, info, st);
}

// H == nullptr: factorisation only (P S = L U), no right-hand sides.
wpccc_status launch_solve(int N, int batch, double2* S, double2* H, int* ipiv, int* info, cudaStream_t st) {
    return lu_launch<double>(N, batch, S, S, H, ipiv, info, st);
}

}  // namespace wpccc

using namespace wpccc;

extern "C" wpccc_status wpccc_solve(int N, int batch, void* S, void* H, int* ipiv, int* info, int precision_mode,
                                    void* stream) {
    if (N < 1 || N > WPCCC_NMAX) return fail(WPCCC_EINVAL, "wpccc_solve: N out of range 1..WPCCC_NMAX");
    if (batch < 0) return fail(WPCCC_EINVAL, "wpccc_solve: batch < 0");
    if (batch > 0 && (!S || !H || !ipiv || !info)) return fail(WPCCC_EINVAL, "wpccc_solve: null pointer");
    if (precision_mode != 0) return fail(WPCCC_EUNSUPPORTED, "wpccc_solve: only precision_mode 0 (FP64)");
    return launch_solve(N, batch, static_cast<double2*>(S), static_cast<double2*>(H), ipiv, info,
                        static_cast<cudaStream_t>(stream));
}
