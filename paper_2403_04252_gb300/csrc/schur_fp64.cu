// The FP64 Schur form's rank-N_T update C = I - K^+ K on the 5th-generation tensor cores, to more than FP64's
// accuracy in norm (I - K^+ K is of order 1, so its small elements need no more).
//
// With X[m][2t] = Re K[t][m], X[m][2t+1] = Im K[t][m] and Y[m][2t] = Im K[t][m], Y[m][2t+1] = -Re K[t][m],
//   (K^+ K)_re[m][n] = sum_k X[m][k] X[n][k],   (K^+ K)_im[m][n] = sum_k X[m][k] Y[n][k],
// a real contraction over k = 2 t + (0, 1) whose rows are written once as eight digits of seven bits
// (k_schur_digits; the representation of mol_fp64.cu, windows of 512 k) and multiplied by k_schur_f64tc, both operands
// by TMA.  On the CUDA cores the update takes 4 N_P^2 N_T FP64 flops of the factorisation's 4 N_P^2 N_T + (4/3) N_P^3 at two
// FMAs per clock per SM: 22 of 30 us per p + H position (N_T = N_P = 190).  Factorisation of 672 such positions, update
// on the CUDA cores -> here: 34.6 -> 15.5 ms; N = 572, 288 positions: 53.7 -> 21.2 ms; N_T = 59, N_P = 50: 0.37 -> 0.27 ms.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "f64_digits.cuh"
#include "wpccc_internal.cuh"

namespace wpccc {

constexpr int SD_DRAIN_WARPS = 8;               // two per TMEM lane quarter, 16 columns each
constexpr int SD_MMA_WARP = SD_DRAIN_WARPS, SD_TMA_WARP = SD_DRAIN_WARPS + 1;
constexpr int SD_THREADS = (SD_TMA_WARP + 1) * 32;
constexpr int SD_A_TILE = F64_M * 64;           // bytes of one digit of the A tile
constexpr int SD_STAGE = F64_SL * (SD_A_TILE + F64_B_TILE);   // 80 KB
constexpr int SD_STAGES = 2;

// Scratch of one position: digit planes [8][2 N_P][KP] bf16 (X rows, then Y rows), scale exponents [windows][N_P].
struct SchurDigits {
    int NP2, KP, nwin;
    size_t ex_off, bytes;
};
static SchurDigits sd_layout(int N, int N_T) {
    SchurDigits L;
    L.NP2 = 2 * (N - N_T);
    L.KP = (2 * N_T + F64_K - 1) / F64_K * F64_K;
    L.nwin = (L.KP + F64_WIN - 1) / F64_WIN;
    L.ex_off = ((size_t)F64_SL * L.NP2 * L.KP * 2 + 255) / 256 * 256;
    L.bytes = (L.ex_off + (size_t)L.nwin * (N - N_T) * sizeof(int) + 255) / 256 * 256;
    return L;
}

// A warp per (projectile state m, window): the digits of X[m] and Y[m], four target states per lane and load.
__global__ void __launch_bounds__(128) k_schur_digits(int N, int N_T, const double2* __restrict__ Sall,
                                                      char* __restrict__ scr, size_t stride, int KP, size_t ex_off) {
    const int NP = N - N_T, lane = threadIdx.x & 31, w = blockIdx.y, e = blockIdx.z;
    const int m = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (m >= NP) return;
    const double2* col = Sall + (size_t)e * N * N + (size_t)(N_T + m) * N;   // K[.][m]
    char* base = scr + (size_t)e * stride;
    __nv_bfloat16* pl = reinterpret_cast<__nv_bfloat16*>(base);
    const size_t plane = (size_t)2 * NP * KP;
    constexpr int Q = F64_WIN / 256;
    double2 z[4 * Q];
    int hm = 0;
#pragma unroll
    for (int j = 0; j < Q; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int t = w * (F64_WIN / 2) + 128 * j + 4 * lane + k;
            z[4 * j + k] = t < N_T ? col[t] : make_double2(0.0, 0.0);
            hm = max(hm, max(abs_hi(z[4 * j + k].x), abs_hi(z[4 * j + k].y)));
        }
    const int E = f64_exponent(__reduce_max_sync(0xffffffffu, hm), F64_MARGIN), E1 = E + 1023;
    if (lane == 0) reinterpret_cast<int*>(base + ex_off)[(size_t)w * NP + m] = E;
#pragma unroll
    for (int j = 0; j < Q; ++j) {
        const int k0 = w * F64_WIN + 256 * j + 8 * lane;
        if (k0 >= KP) continue;
        uint32_t x[4][F64_SL], y[4][F64_SL];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double2 a = z[4 * j + k];
            const uint64_t re = f64_fix(a.x, E1), im = f64_fix(a.y, E1);
            f64_digits(re, im, x[k]);
            f64_digits(im, f64_fix(-a.x, E1), y[k]);
        }
#pragma unroll
        for (int i = 0; i < F64_SL; ++i) {
            *reinterpret_cast<uint4*>(pl + i * plane + (size_t)m * KP + k0) = make_uint4(x[0][i], x[1][i], x[2][i], x[3][i]);
            *reinterpret_cast<uint4*>(pl + i * plane + (size_t)(NP + m) * KP + k0) = make_uint4(y[0][i], y[1][i], y[2][i], y[3][i]);
        }
    }
}

struct SdMaps {
    CUtensorMap a, b;   // digit planes with box heights 128 and 32
};

struct SdArgs {
    int N, N_T, NP, KP, nwin;
    const char* scr;
    size_t stride, ex_off;
    double2* S;             // [nev][N][N]: C into the projectile block's lower triangle
    int* err;
    long wait_limit;
};

// Tiles of 128 rows (of X) by 32 rows (of X, then of Y) that touch the lower triangle.
static __host__ __device__ inline int sd_tiles_of(int a, int NP) { return 2 * ((min(NP, a + F64_M) + F64_N - 1) / F64_N); }

__global__ void __launch_bounds__(SD_THREADS, 1) k_schur_f64tc(const __grid_constant__ SdMaps maps, SdArgs A) {
    extern __shared__ __align__(1024) unsigned char sd_smem_raw[];
    unsigned char* sm = sd_smem_raw + ((1024 - (smem_u32(sd_smem_raw) & 1023)) & 1023);
    __shared__ uint64_t s_bars[2 * SD_STAGES + 2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, e = blockIdx.y;
    int a0 = 0, tile = blockIdx.x;
    while (tile >= sd_tiles_of(a0, A.NP)) {
        tile -= sd_tiles_of(a0, A.NP);
        a0 += F64_M;
    }
    const int per = sd_tiles_of(a0, A.NP) / 2, half = tile >= per;
    const int n0 = (tile - (half ? per : 0)) * F64_N, b0 = half * A.NP + n0;   // first projectile column, first plane row
    const uint32_t full0 = smem_u32(s_bars), done0 = full0 + 8 * SD_STAGES, accf = done0 + 8 * SD_STAGES, acce = accf + 8;
    if (tid == 0) {
        s_abort = 0;
        for (int s = 0; s < SD_STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(done0 + 8 * s, 1);
        }
        mbar_init(accf, 1);
        mbar_init(acce, SD_DRAIN_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)),
                     "r"(F64_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    volatile int* abort_flag = &s_abort;
    const int nk = A.KP / F64_K;

    if (warp == SD_TMA_WARP) {
        if (lane == 0) {
            int issued = 0;
            for (; issued < nk; ++issued) {
                const int s = issued % SD_STAGES, kp = issued - SD_STAGES;
                if (kp >= 0 && !mbar_wait(done0 + 8 * s, (kp / SD_STAGES) & 1, abort_flag, A.err, 41, A.wait_limit)) break;
                const uint32_t st = smem_u32(sm) + (uint32_t)(s * SD_STAGE), bar = full0 + 8 * s;
                mbar_arrive_tx(bar, SD_STAGE);
                for (int i = 0; i < F64_SL; ++i) {
                    tma_load_3d(st + i * SD_A_TILE, &maps.a, issued * F64_K, i * 2 * A.NP + a0, e, bar);
                    tma_load_3d(st + F64_SL * SD_A_TILE + i * F64_B_TILE, &maps.b, issued * F64_K, i * 2 * A.NP + b0, e, bar);
                }
            }
            // every copy issued has landed before the CTA exits
            for (int k = issued > SD_STAGES ? issued - SD_STAGES : 0; k < issued; ++k)
                for (long it = 0; it < TC_WAIT_LIMIT && !mbar_try(full0 + 8 * (k % SD_STAGES), (k / SD_STAGES) & 1); ++it) {
                }
        }
    } else if (warp == SD_MMA_WARP) {
        if (lane == 0) {
            bool ok = true, ready = false;
            int issued = 0;
            auto wait = [&](uint32_t bar, uint32_t par, int code) {
                return mbar_test(bar, par) || mbar_wait(bar, par, abort_flag, A.err, code, A.wait_limit);
            };
            for (int k = 0; k < nk && ok; ++k) {
                const int s = k % SD_STAGES;
                const bool fresh = k % F64_WCH == 0;
                if (!ready) ok = wait(full0 + 8 * s, (k / SD_STAGES) & 1, 42);
                if (ok && fresh && k > 0) ok = wait(acce, (k / F64_WCH - 1) & 1, 43);
                if (!ok) break;
                tc_fence_after();
                const uint32_t st = smem_u32(sm) + (uint32_t)(s * SD_STAGE);
                f64_mma_chunk(tmem, sw64_desc(st), sw64_desc(st + F64_SL * SD_A_TILE), SD_A_TILE >> 4, fresh, [&] {
                    ready = k + 1 < nk && mbar_test(full0 + 8 * ((k + 1) % SD_STAGES), ((k + 1) / SD_STAGES) & 1);
                });
                tc_commit(done0 + 8 * s);
                issued = k + 1;
                if (k % F64_WCH == F64_WCH - 1 || k == nk - 1) tc_commit(accf);
            }
            // the MMAs issued complete before the tensor memory is released
            if (issued > 0)
                for (long it = 0; it < TC_WAIT_LIMIT &&
                                  !mbar_try(done0 + 8 * ((issued - 1) % SD_STAGES), ((issued - 1) / SD_STAGES) & 1); ++it) {
                }
        }
    } else {
        // drain: TMEM lanes 32 qd .. 32 qd + 31 (rows m), 16 columns from col0
        const int qd = warp & 3, col0 = (warp >> 2) * 16, m = a0 + qd * 32 + lane;
        const int* ex = reinterpret_cast<const int*>(A.scr + (size_t)e * A.stride + A.ex_off);
        double acc[16];
        float low[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            acc[k] = 0.0;
            low[k] = 0.f;
        }
        bool ok = true;
        for (int j = 0; j < A.nwin && ok; ++j) {
            const int Em = m < A.NP ? ex[(size_t)j * A.NP + m] : F64_EMIN;
            const int nn = n0 + col0 + (lane & 15), En = nn < A.NP ? ex[(size_t)j * A.NP + nn] : F64_EMIN;
            ok = mbar_wait_warp(accf, j & 1, abort_flag, A.err, 44, A.wait_limit);
            if (!ok) break;
            tc_fence_after();
            const uint32_t base = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)col0;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                float v[F64_LEV][4];
#pragma unroll
                for (int L = 0; L < F64_LEV; ++L) tmem_ld4(base + (uint32_t)(L * F64_N + 4 * g), v[L]);
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    long long T;
                    uint32_t low19;
                    f64_levels(v, u, T, low19);
                    f64_accumulate(acc[4 * g + u], low[4 * g + u], T, low19, Em + __shfl_sync(0xffffffffu, En, 4 * g + u), F64_UNIT);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce);
        }
        if (ok && m < A.NP) {
            double2* S = A.S + (size_t)e * A.N * A.N;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int n = n0 + col0 + k;
                if (n >= A.NP || n > m) continue;
                const double c = f64_total(acc[k], low[k], F64_UNIT);
                double* p = reinterpret_cast<double*>(S + (size_t)(A.N_T + m) + (size_t)(A.N_T + n) * A.N);
                if (half) p[1] = -c;
                else p[0] = (m == n ? 1.0 : 0.0) - c;
            }
        }
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(F64_TMEM_COLS));
    }
}

// From 16 target states on (one 32-term chunk): a smaller update costs less than two more launches (N_T = 2, N_P = 52:
// 1.53 ms without, 1.76 with).  No rule on N_P: N_P = 2, N_T = 57 takes 0.047 ms without, 0.037 with.
bool schur_fp64_tc_applicable(const wpccc_basis_s* B, size_t scratch_per_eval) {
    if (!encode_fn() || B->n_centres != 2 || !B->tc_err || B->N_T < F64_K / 2) return false;
    return sd_layout(B->N, B->N_T).bytes <= scratch_per_eval;
}

wpccc_status launch_schur_factor_fp64_tc(wpccc_basis_s* B, int nev, double2* S, int* info, void* scratch,
                                         size_t scratch_per_eval, cudaStream_t st) {
    if (nev == 0) return WPCCC_OK;
    const int N = B->N, N_T = B->N_T, NP = N - N_T;
    const SchurDigits L = sd_layout(N, N_T);
    if (L.bytes > scratch_per_eval || (uintptr_t)scratch % 16 != 0 || !B->tc_err)
        return fail(WPCCC_EINVAL, "FP64 tensor-core Schur update: scratch");
    k_schur_digits<<<dim3((NP + 3) / 4, L.nwin, nev), 128, 0, st>>>(N, N_T, S, static_cast<char*>(scratch), L.bytes, L.KP,
                                                                    L.ex_off);
    WPCCC_CHECK_LAUNCH("k_schur_digits");
    SdMaps maps;
    const cuuint64_t dims[3] = {(cuuint64_t)L.KP, (cuuint64_t)F64_SL * L.NP2, (cuuint64_t)nev};
    const cuuint64_t strides[2] = {(cuuint64_t)L.KP * 2, (cuuint64_t)L.bytes};
    const cuuint32_t estr[3] = {1, 1, 1};
    const cuuint32_t boxa[3] = {(cuuint32_t)F64_K, (cuuint32_t)F64_M, 1}, boxb[3] = {(cuuint32_t)F64_K, (cuuint32_t)F64_N, 1};
    for (int k = 0; k < 2; ++k) {
        CUresult r = encode_fn()(k == 0 ? &maps.a : &maps.b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, scratch, dims, strides,
                                 k == 0 ? boxa : boxb, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return fail(WPCCC_ECUDA, "cuTensorMapEncodeTiled failed for the Schur digit planes");
    }
    SdArgs a;
    a.N = N;
    a.N_T = N_T;
    a.NP = NP;
    a.KP = L.KP;
    a.nwin = L.nwin;
    a.scr = static_cast<const char*>(scratch);
    a.stride = L.bytes;
    a.ex_off = L.ex_off;
    a.S = S;
    a.err = B->tc_err;
    a.wait_limit = B->wait_polls;
    int tiles = 0;
    for (int a0 = 0; a0 < NP; a0 += F64_M) tiles += sd_tiles_of(a0, NP);
    const size_t smem = 1024 + (size_t)SD_STAGES * SD_STAGE;
    WPCCC_CUDA(cudaFuncSetAttribute(k_schur_f64tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_schur_f64tc<<<dim3(tiles, nev), SD_THREADS, smem, st>>>(maps, a);
    WPCCC_CHECK_LAUNCH("k_schur_f64tc");
    return launch_schur_cholesky(N, N_T, nev, S, info, st);
}

}  // namespace wpccc
