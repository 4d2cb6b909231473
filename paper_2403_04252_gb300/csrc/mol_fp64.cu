// Eq. 9 contraction of the FP64 form on the 5th-generation tensor cores, at FP64's accuracy element by element.
//
// For one row tile (target states of one molecular-frame projection q') the two-centre integrals are
//   X_K[i][c] = sum_g (A_T r_T)[i][g] b[c][g],   X_Q[i][c] = sum_g (A_T r_T V_T)[i][g] b[c][g],
//   b[(c, re/im)][g] = re/im(W_{|q_c - q'|}(g) / r_T(g)) A_P[c][g],
// a real contraction over the quadrature nodes g of M = 128 table rows and N = 32 generated rows
// (16 half columns x re/im) per thread block.
//
// Representation.  Per window of 512 nodes (fewer far from the target, see below) every row of both operands is written in fixed point against
// the power of two above the row's largest |value| of the window, x = X 2^(E - 55) with X rounded to an integer
// (|X| < 2^55), and X in eight balanced digits of seven bits, X = sum_i k_i 2^(49 - 7 i), k_i in [-64, 63], each an
// exact bf16 number k_i 2^(-7 i) (the error-free slicing of Ozaki, Ogita, Oishi and Rump, with a fixed grid per
// window).  Products of digits i + j = L form level L; levels 0..8 (43 products) have an FP32 accumulator each, whose
// sum over a window is an integer of at most 8 x 2^12 x 512 = 2^24 units, so every accumulation is exact in any
// order.  Levels >= 9 are dropped: below 2^-60 of the window's largest product.  Per window the levels are put
// together as one 51-bit and one 19-bit integer and added to the FP64 running sums (one FP64 FMA; the low bits go
// to an FP32 sum of weight 2^-61).  The generated values are rounded once to FP64 as W A_P, as in the CUDA-core
// contraction.
//
// Accuracy.  A window's rounding is relative to the product of its rows' largest values.  In 2-norm the off-diagonal
// blocks of two-centre p + H err by 1e-17 to 2e-17 (against long double, |z| <= 12), the chain of G multiply-adds by 8e-17
// to 1.3e-15.  A small element whose rows peak at different nuclei is far below that product, so the nodes' order, the
// windows' length and exact power-of-two scales keep the two together (f64_order.cuh): element by element the error
// stays within what the chain leaves (its comment has the figures).  The shorter windows cost a drain each, with two FP64 operations per
// result: 33, 43, 67 and 125 us per p + H position with windows of 512, 128, 64 and 32 nodes (24 positions); 21 positions
// over |z| <= 20 take 1.3 to 1.4 ms a call, 1.20 with windows of 512 nodes throughout.
//
// What bounds it.  The FP64 pipe of this part does two FMAs per clock per SM, and the CUDA-core contraction takes
// five FP64 operations per (target state, half column, node): 581 us per p + H position (N = 380, 2304 nodes).  Here
// the FP64 pipe forms one product per generated element and two operations per result and window; the MMAs set
// the pace (tensor pipe 59 % busy; a 128-row tile holds 22 to 100 rows of p + H).  Measured, 24 p + H positions near the
// target: 33 us per position, of which 18 us are the tensor cores' own time, plus 8 us for the operands (k_f64_slices).
// The MMA queue is short, so the issuing thread's scalar work between two chunks shows in full: carrying the ring
// positions along and testing the next chunk's barriers early took 2360 -> 1750 cycles per chunk (1281 of MMAs).

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "f64_digits.cuh"
#include "f64_order.cuh"
#include "geometry.cuh"
#include "wpccc_internal.cuh"

namespace wpccc {

constexpr int F64_HALF = F64_N / 2;             // half columns per CTA
constexpr int F64_PROD_WARPS = 8;               // producers: a thread per (half column, node pair)
constexpr int F64_DRAIN_WARPS = 8;              // two per TMEM lane quarter, 16 columns each
constexpr int F64_MMA_WARP = F64_PROD_WARPS + F64_DRAIN_WARPS;
constexpr int F64_TMA_WARP = F64_MMA_WARP + 1;
constexpr int F64_THREADS = (F64_TMA_WARP + 1) * 32;
constexpr int F64_GSTAGE = F64_SL * F64_B_TILE; // 16 KB
constexpr int F64_GSTAGES = 4;
constexpr int F64_RING = 160 * 1024;            // table ring: as many chunks as the tile's height allows
constexpr int F64_TSTAGES_MAX = 8;
constexpr int F64_DONE = 8;                     // ring of "MMAs of a chunk completed" barriers (>= every other ring)
constexpr int F64_SPLIT = 4;                    // blocks of k_f64_slices per span of 512 nodes

// ---------------------------------------------------------------------------
// k_f64_slices: the operands of the contraction from the FP64 node tables.
// F64_SPLIT blocks per (span of 512 nodes, position): a warp per projectile half column (A_P and the scale exponents of
// its generated rows), then a warp per (target radial, |m|) (digits of A_T r_T and A_T r_T V_T; the rows of m and
// -m differ by the sign (-1)^m).  Lane: nodes 4 lane .. 4 lane + 3 and 128, 256, 384 further.
// ---------------------------------------------------------------------------
struct F64SliceArgs {
    const EvalDesc* ev;
    double kappa;
    int G, Gp, nradT, nradP, nlqT, nd, n_half, tc_rows, nwin, n_items, qmaxT;
    const int* items;       // [n_items][7]: radial, (l, |m|) index, 1 when m odd, row of +m, row of -m (or -1), sizes of their tiles
    const int* halves;      // [n_half][3]: radial, (l, q) index, q
    char* node;             // node tables; the layout's offsets in bytes from each position's start
    size_t node_bytes, pl_off, ea_off, eb_off, ap_off, w2_off, r_off;
};

static __device__ __forceinline__ void load4(const double* __restrict__ p, int g, int G, bool vec, double v[4]) {
    if (vec && g + 3 < G) {
        const double2 a = *reinterpret_cast<const double2*>(p + g), b = *reinterpret_cast<const double2*>(p + g + 2);
        v[0] = a.x;
        v[1] = a.y;
        v[2] = b.x;
        v[3] = b.y;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = g + k < G ? p[g + k] : 0.0;
    }
}

// FULL: one window per span (wch = 16); else wch chunks of 32 nodes per window.
template <bool FULL>
static __device__ __forceinline__ void f64_slices(const F64SliceArgs& A, int wch, double* s_r, double* s_rv, int* s_hw) {
    const int e = blockIdx.y, w = blockIdx.x / F64_SPLIT, part = blockIdx.x % F64_SPLIT, g0 = w * F64_WIN;
    const int tid = threadIdx.x, warp = part * 8 + (tid >> 5), lane = tid & 31;   // warp among the span's
    constexpr int Q = F64_WIN / 128, NW = FULL ? 1 : Q;   // node quads per lane; windows that they lie in
    // m[j] <- the largest m over the window of the lane's quad j
    auto window_max = [&](int (&m)[NW]) {
#pragma unroll
        for (int j = 0; j < NW; ++j) {
            if (FULL || wch == 4) m[j] = __reduce_max_sync(0xffffffffu, m[j]);
            else
                for (int o = 4 * wch; o > 0; o >>= 1) m[j] = max(m[j], __shfl_xor_sync(0xffffffffu, m[j], o));
        }
    };
    // that window, for the one lane that writes it; else -1
    int window[NW];
#pragma unroll
    for (int j = 0; j < NW; ++j) {
        const int g = g0 + 4 * lane + 128 * j, per = FULL ? F64_WIN : wch * F64_K;
        window[j] = g < A.Gp && (g & (per - 1)) == 0 ? g / per : -1;
    }
    char* base = A.node + (size_t)e * A.node_bytes;
    const double* fT = reinterpret_cast<const double*>(base);
    const double* fP = fT + (size_t)A.nradT * A.G;
    const double* thT = fP + (size_t)A.nradP * A.G;
    const double* thP = thT + (size_t)A.nlqT * A.G;
    const bool vec = (A.G & 1) == 0;   // the rows start on 16-byte boundaries
    const double* w2 = reinterpret_cast<const double*>(base + A.w2_off);
    const double* rr = reinterpret_cast<const double*>(base + A.r_off);
    for (int o = tid; o < F64_WIN; o += 256) {
        const int g = g0 + o;
        const bool in = g < A.Gp;
        s_r[o] = in ? rr[g] : 0.0;
        s_rv[o] = in ? rr[A.Gp + g] : 0.0;
        for (int d = 0; d < A.nd; ++d)
            s_hw[d * F64_WIN + o] =
                in ? max(abs_hi(w2[(size_t)(2 * d) * A.Gp + g]), abs_hi(w2[(size_t)(2 * d + 1) * A.Gp + g])) : 0;
    }
    __syncthreads();
    // projectile half columns: A_P, and per d = |q - q'| the scale exponent of W A_P over the window
    double* ap = reinterpret_cast<double*>(base + A.ap_off);
    int* eb = reinterpret_cast<int*>(base + A.eb_off);
    for (int c = warp; c < A.n_half; c += 8 * F64_SPLIT) {
        const double* f = fP + (size_t)A.halves[3 * c] * A.G;
        const double* th = thP + (size_t)A.halves[3 * c + 1] * A.G;
        const int q = A.halves[3 * c + 2];
        int h[F64_WIN / 32];
#pragma unroll
        for (int j = 0; j < F64_WIN / 128; ++j) {
            const int o = 4 * lane + 128 * j, g = g0 + o;
            double fv[4], tv[4];
            load4(f, g, A.G, vec, fv);
            load4(th, g, A.G, vec, tv);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                fv[k] *= tv[k];
                h[4 * j + k] = abs_hi(fv[k]);
            }
            if (g < A.Gp) {
                *reinterpret_cast<double2*>(ap + (size_t)c * A.Gp + g) = make_double2(fv[0], fv[1]);
                *reinterpret_cast<double2*>(ap + (size_t)c * A.Gp + g + 2) = make_double2(fv[2], fv[3]);
            }
        }
        const int dlo = max(0, q - A.qmaxT), dhi = min(A.nd - 1, q + A.qmaxT);
        for (int d = dlo; d <= dhi; ++d) {
            int m[NW] = {};
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                const int4 hw = *reinterpret_cast<const int4*>(s_hw + d * F64_WIN + 4 * lane + 128 * j);
                const int hv[4] = {hw.x, hw.y, hw.z, hw.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int a = h[4 * j + k], b = hv[k];
                    // zero and denormal factors leave the window's scale alone; a non-finite one marks the row (the sum of
                    // two high words passes 2^31 from a product of 4 on: unsigned)
                    const uint32_t ab = (uint32_t)a + (uint32_t)b;
                    const int p = max(a, b) >= 0x7FF00000 ? 0x7FF00000
                                  : min(a, b) < (1 << 20) || ab < (1023u << 20) ? 0 : (int)min(ab - (1023u << 20), 0x7FEFFFFFu);
                    m[FULL ? 0 : j] = max(m[FULL ? 0 : j], p);
                }
            }
            window_max(m);
#pragma unroll
            for (int j = 0; j < NW; ++j)
                if (window[j] >= 0) eb[((size_t)c * A.nd + d) * A.nwin + window[j]] = f64_exponent(m[j], F64_MARGIN2);
        }
    }
    // target rows
    __nv_bfloat16* pl = reinterpret_cast<__nv_bfloat16*>(base + A.pl_off);
    int* ea = reinterpret_cast<int*>(base + A.ea_off);
    const size_t plane = (size_t)A.tc_rows * A.Gp;
    for (int it = warp; it < A.n_items; it += 8 * F64_SPLIT) {
        const int* I = A.items + 7 * it;
        const double* f = fT + (size_t)I[0] * A.G;
        const double* th = thT + (size_t)I[1] * A.G;
        const bool odd = I[2] != 0;
        const int rp = I[3], rn = I[4], ts = I[5], tsn = I[6];
        double t[4 * Q];
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            double fv[4], tv[4];
            load4(f, g0 + 4 * lane + 128 * j, A.G, vec, fv);
            load4(th, g0 + 4 * lane + 128 * j, A.G, vec, tv);
#pragma unroll
            for (int k = 0; k < 4; ++k) t[4 * j + k] = fv[k] * tv[k];
        }
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const double* sr = v == 0 ? s_r : s_rv;
            double x[4 * Q];
            int m[NW] = {};
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                const double2 ra = *reinterpret_cast<const double2*>(sr + 4 * lane + 128 * j),
                              rb = *reinterpret_cast<const double2*>(sr + 4 * lane + 128 * j + 2);
                x[4 * j] = t[4 * j] * ra.x;
                x[4 * j + 1] = t[4 * j + 1] * ra.y;
                x[4 * j + 2] = t[4 * j + 2] * rb.x;
                x[4 * j + 3] = t[4 * j + 3] * rb.y;
#pragma unroll
                for (int k = 0; k < 4; ++k) m[FULL ? 0 : j] = max(m[FULL ? 0 : j], abs_hi(x[4 * j + k]));
            }
            window_max(m);
            const int r1 = rp + v * ts, r2 = rn + v * tsn;
            int E[NW];
#pragma unroll
            for (int j = 0; j < NW; ++j) {
                E[j] = f64_exponent(m[j], F64_MARGIN);
                if (window[j] < 0) continue;
                ea[(size_t)window[j] * A.tc_rows + r1] = E[j];
                if (rn >= 0) ea[(size_t)window[j] * A.tc_rows + r2] = E[j];
            }
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                const int g = g0 + 4 * lane + 128 * j, E1 = E[FULL ? 0 : j] + 1023;
                if (g >= A.Gp) continue;
                uint32_t d0[F64_SL], d1[F64_SL];
                f64_digits(f64_fix(x[4 * j], E1), f64_fix(x[4 * j + 1], E1), d0);
                f64_digits(f64_fix(x[4 * j + 2], E1), f64_fix(x[4 * j + 3], E1), d1);
#pragma unroll
                for (int i = 0; i < F64_SL; ++i)
                    *reinterpret_cast<uint2*>(pl + i * plane + (size_t)r1 * A.Gp + g) = make_uint2(d0[i], d1[i]);
                if (rn >= 0) {
                    if (odd) {
                        f64_digits(f64_fix(-x[4 * j], E1), f64_fix(-x[4 * j + 1], E1), d0);
                        f64_digits(f64_fix(-x[4 * j + 2], E1), f64_fix(-x[4 * j + 3], E1), d1);
                    }
#pragma unroll
                    for (int i = 0; i < F64_SL; ++i)
                        *reinterpret_cast<uint2*>(pl + i * plane + (size_t)r2 * A.Gp + g) = make_uint2(d0[i], d1[i]);
                }
            }
        }
    }
}

__global__ void __launch_bounds__(256) k_f64_slices(F64SliceArgs A) {
    __shared__ __align__(16) double s_r[F64_WIN], s_rv[F64_WIN];
    extern __shared__ int s_hw[];   // [nd][F64_WIN]: high word of max(|re|, |im|) of W / r_T
    const EvalDesc& p = A.ev[blockIdx.y];
    const int wch = f64_window_chunks(A.Gp, __dmul_rn(A.kappa, dist_R(p.b, p.z)));
    if (wch * F64_K == F64_WIN) f64_slices<true>(A, wch, s_r, s_rv, s_hw);
    else f64_slices<false>(A, wch, s_r, s_rv, s_hw);
}

// ---------------------------------------------------------------------------
// k_mol_f64tc: the contraction
// ---------------------------------------------------------------------------
struct F64Maps {
    CUtensorMap m[F64_M / 32];   // digit planes with box heights 32, 64, 96 and 128 rows
};

struct F64Args {
    const EvalDesc* ev;
    double kappa;
    int Gp, N_T, n_half, nk, nwin, nd, n_ntiles, tc_rows, qg_max;
    const int *qg_off, *qg_q, *qg_rows, *half_q;
    const char* node;
    size_t node_bytes, ea_off, eb_off, ap_off, w2_off;
    double* mol;            // [nev][2][N_T][n_half] complex
    int* err;
    long wait_limit;
};

__global__ void __launch_bounds__(F64_THREADS, 1) k_mol_f64tc(const __grid_constant__ F64Maps maps, F64Args A) {
    extern __shared__ __align__(1024) unsigned char f64_smem_raw[];
    unsigned char* sm = f64_smem_raw + ((1024 - (smem_u32(f64_smem_raw) & 1023)) & 1023);
    unsigned char* gsm = sm + F64_RING;
    __shared__ uint64_t s_bars[F64_TSTAGES_MAX + F64_GSTAGES + F64_DONE + 2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ntile = blockIdx.x % A.n_ntiles, tile = blockIdx.x / A.n_ntiles, e = blockIdx.y;
    const int row0 = A.qg_off[tile], ns = (A.qg_off[tile + 1] - row0) / 2;
    const int qp = A.qg_q[tile];
    const int box = (2 * ns + 31) / 32;                       // table box height, in 32-row units
    const uint32_t a_tile = (uint32_t)box * 32 * 64;          // bytes of one digit of the table tile
    const uint32_t tstage = F64_SL * a_tile;
    const int nst = min(F64_TSTAGES_MAX, (int)(F64_RING / tstage));
    const int c0 = ntile * F64_HALF;
    // tfull (TMA), gfull (producers), done (MMA commit: frees the table stage and the generated stage of a chunk), accf
    // (MMA commit), acce (drain).  A slot of `done` is reused after eight chunks: by then the TMA thread and every
    // producer have waited for its previous phase, since they issue a chunk only after that.
    const uint32_t tfull0 = smem_u32(s_bars), gfull0 = tfull0 + 8 * F64_TSTAGES_MAX, done0 = gfull0 + 8 * F64_GSTAGES,
                   accf = done0 + 8 * F64_DONE, acce = accf + 8;
    if (tid == 0) {
        s_abort = 0;
        for (int s = 0; s < F64_TSTAGES_MAX; ++s) mbar_init(tfull0 + 8 * s, 1);
        for (int s = 0; s < F64_GSTAGES; ++s) mbar_init(gfull0 + 8 * s, F64_PROD_WARPS);
        for (int s = 0; s < F64_DONE; ++s) mbar_init(done0 + 8 * s, 1);
        mbar_init(accf, 1);
        mbar_init(acce, F64_DRAIN_WARPS);
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
    const char* nb = A.node + (size_t)e * A.node_bytes;
    const int nk = A.nk;
    const double kR = __dmul_rn(A.kappa, dist_R(A.ev[e].b, A.ev[e].z));
    const int wch = f64_window_chunks(A.Gp, kR), wlog = 31 - __clz(wch);

    if (warp == F64_TMA_WARP) {
        // ---- TMA issue (one thread): the table tiles chunk by chunk into their ring
        if (lane == 0) {
            const CUtensorMap* tmap = &maps.m[box - 1];
            auto issue = [&](int k) {
                const int s = k % nst;
                const uint32_t st = smem_u32(sm) + (uint32_t)s * tstage, bar = tfull0 + 8 * s;
                mbar_arrive_tx(bar, tstage);
                for (int i = 0; i < F64_SL; ++i)
                    tma_load_3d(st + i * a_tile, tmap, k * F64_K, i * A.tc_rows + row0, e, bar);
            };
            int issued = 0;
            for (; issued < nk; ++issued) {
                const int kp = issued - nst;
                if (kp >= 0 &&
                    !mbar_wait(done0 + 8 * (kp % F64_DONE), (kp / F64_DONE) & 1, abort_flag, A.err, 31, A.wait_limit))
                    break;
                issue(issued);
            }
            // every copy issued has landed before the CTA exits (at once on the normal path, bounded otherwise)
            for (int k = issued > nst ? issued - nst : 0; k < issued; ++k)
                for (long it = 0; it < TC_WAIT_LIMIT && !mbar_try(tfull0 + 8 * (k % nst), (k / nst) & 1); ++it) {
                }
        }
    } else if (warp == F64_MMA_WARP) {
        // ---- MMA issue (one thread)
        if (lane == 0) {
            bool ok = true;
            int issued = 0;
            // Ring positions and phases are carried along instead of divided out, and the next chunk's barriers are tested
            // between this chunk's two K steps: the MMA queue is short, so scalar latency between two chunks' MMAs
            // leaves the tensor cores idle.
            uint32_t ts = 0, tph = 0, gs = 0, gph = 0, dsl = 0;
            const uint64_t da0 = sw64_desc(smem_u32(sm)), db0 = sw64_desc(smem_u32(gsm));
            auto wait = [&](uint32_t bar, uint32_t par, int code) {
                return mbar_test(bar, par) || mbar_wait(bar, par, abort_flag, A.err, code, A.wait_limit);
            };
            bool ready = false;
            for (int k = 0; k < nk && ok; ++k) {
                const bool fresh = (k & (wch - 1)) == 0;   // the window's first products overwrite the accumulators
                if (!ready) ok = wait(tfull0 + 8 * ts, tph, 32) && wait(gfull0 + 8 * gs, gph, 33);
                if (ok && fresh && k > 0) ok = wait(acce, ((k >> wlog) - 1) & 1, 34);
                if (!ok) break;
                tc_fence_after();
                const uint64_t da = da0 + (uint64_t)(ts * (tstage >> 4)), db = db0 + (uint64_t)(gs * (F64_GSTAGE >> 4));
                ts = ts + 1 == (uint32_t)nst ? 0 : ts + 1;
                tph ^= ts == 0;
                gs = (gs + 1) % F64_GSTAGES;
                gph ^= gs == 0;
                f64_mma_chunk(tmem, da, db, a_tile >> 4, fresh, [&] {
                    ready = k + 1 < nk && mbar_test(tfull0 + 8 * ts, tph) && mbar_test(gfull0 + 8 * gs, gph);
                });
                tc_commit(done0 + 8 * dsl);
                dsl = (dsl + 1) % F64_DONE;
                issued = k + 1;
                if ((k & (wch - 1)) == wch - 1 || k == nk - 1) tc_commit(accf);
            }
            // the MMAs issued complete before the tensor memory is released
            if (issued > 0)
                for (long it = 0; it < TC_WAIT_LIMIT && !mbar_try(done0 + 8 * ((issued - 1) % F64_DONE), ((issued - 1) / F64_DONE) & 1); ++it) {
                }
        }
    } else if (warp >= F64_PROD_WARPS) {
        // ---- drain: TMEM lanes 32 qd .. 32 qd + 31 (table rows), 16 columns from col0 (generated rows)
        const int dw = warp - F64_PROD_WARPS, qd = warp & 3, col0 = (dw >> 2) * 16;
        const int lrow = qd * 32 + lane;
        const bool live = qd * 32 < 2 * ns;
        const int* ea = reinterpret_cast<const int*>(nb + A.ea_off);
        const int* eb = reinterpret_cast<const int*>(nb + A.eb_off);
        // lanes 0..7: scale exponents of this warp's eight half columns
        size_t ebo = 0;
        bool ebv = false;
        if (lane < 8 && c0 + col0 / 2 + lane < A.n_half) {
            const int c = c0 + col0 / 2 + lane, d = abs(A.half_q[c] - qp);
            ebo = ((size_t)c * A.nd + d) * A.nwin;
            ebv = true;
        }
        double acc[16];
        float low[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            acc[k] = 0.0;
            low[k] = 0.f;
        }
        bool ok = true;
        const int nwin = (nk + wch - 1) >> wlog;
        // the low parts' unit follows the largest scales of the element's two rows
        int ua = F64_EMIN, ub = F64_EMIN;
        for (int j = 0; j < nwin; ++j) {
            if (lrow < 2 * ns) ua = max(ua, ea[(size_t)j * A.tc_rows + row0 + lrow]);
            if (ebv) ub = max(ub, eb[ebo + j]);
        }
        ua = F64_UNIT - max(-500, min(ua, 500));
        ub = -max(-500, min(ub, 500));
        for (int j = 0; j < nwin && ok; ++j) {
            const int Ea = lrow < 2 * ns ? ea[(size_t)j * A.tc_rows + row0 + lrow] : F64_EMIN;
            const int Eb = ebv ? eb[ebo + j] : F64_EMIN;
            ok = mbar_wait_warp(accf, j & 1, abort_flag, A.err, 35, A.wait_limit);
            if (!ok) break;
            tc_fence_after();
            // first the nine levels of each element are put together; then the accumulators are free for the next
            // window, and the FP64 work on T overlaps its MMAs
            long long T[16];
            uint32_t low19[16];
            if (live) {
                const uint32_t base = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)col0;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    float v[F64_LEV][4];
#pragma unroll
                    for (int L = 0; L < F64_LEV; ++L) tmem_ld4(base + (uint32_t)(L * F64_N + 4 * g), v[L]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        f64_levels(v, u, T[4 * g + u], low19[4 * g + u]);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce);
            if (live) {
#pragma unroll
                for (int k = 0; k < 16; ++k)
                    f64_accumulate(acc[k], low[k], T[k], low19[k], Ea + __shfl_sync(0xffffffffu, Eb, k >> 1),
                                   ua + __shfl_sync(0xffffffffu, ub, k >> 1));
            }
        }
        // results: row lrow of D is A_T row lrow of the tile (overlap K) or, from ns on, its A_T V_T row (Q)
        if (ok) {
            const int x = lrow < ns ? 0 : 1;
            const int i = lrow < 2 * ns ? A.qg_rows[tile * A.qg_max + (lrow < ns ? lrow : lrow - ns)] : 0;
            const size_t plane = (size_t)A.N_T * A.n_half;
            double2* out = reinterpret_cast<double2*>(A.mol) + (size_t)e * 2 * plane + (size_t)x * plane + (size_t)i * A.n_half;
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const int c = c0 + (col0 + k) / 2, unit = ua + __shfl_sync(0xffffffffu, ub, k >> 1);
                if (lrow < 2 * ns && c < A.n_half)
                    out[c] = make_double2(f64_total(acc[k], low[k], unit), f64_total(acc[k + 1], low[k + 1], unit));
            }
        }
    } else {
        // ---- producers: thread = (half column, node pair); one FP64 multiplication per element, then an integer shift
        // rounds W A_P to the window's grid.  The next chunk's A_P and W are loaded before this chunk is written.
        const int p = tid & 15, cl = tid >> 4, c = c0 + cl;
        const bool valid = c < A.n_half;
        const int d = valid ? abs(A.half_q[c] - qp) : 0;
        const double* ap = reinterpret_cast<const double*>(nb + A.ap_off) + (size_t)(valid ? c : 0) * A.Gp + 2 * p;
        const double* wr = reinterpret_cast<const double*>(nb + A.w2_off) + (size_t)(2 * d) * A.Gp + 2 * p;
        const double* wi = wr + A.Gp;
        const int* eb = reinterpret_cast<const int*>(nb + A.eb_off) + ((size_t)(valid ? c : 0) * A.nd + d) * A.nwin;
        // row n = 2 cl + re/im of each digit tile: 64 bytes, 16-byte piece at (piece ^ ((n >> 1) & 3))
        const uint32_t off = (uint32_t)(2 * cl) * 64 + (uint32_t)(((p >> 2) ^ (cl & 3)) << 4) + (uint32_t)((p & 3) * 4);
        const uint32_t ro = off + (uint32_t)((cl & 1) * 64), io = off + (uint32_t)((~cl & 1) * 64);
        const double2 zero = make_double2(0.0, 0.0);
        double2 a = valid ? *reinterpret_cast<const double2*>(ap) : zero;
        double2 r = *reinterpret_cast<const double2*>(wr), im = *reinterpret_cast<const double2*>(wi);
        int E = valid ? eb[0] : F64_EMIN;
        bool ok = true;
        for (int k = 0; k < nk && ok; ++k) {
            const int s = k % F64_GSTAGES;
            const int E1 = E + 1023;
            // odd half columns write their imaginary row first: the two half columns of a warp then store to
            // different halves of the 128 bytes of banks
            const double2 w0 = (cl & 1) ? im : r, w1 = (cl & 1) ? r : im, ac = a;
            if (k + 1 < nk) {
                const int g = (k + 1) * F64_K;
                if (valid) {
                    a = *reinterpret_cast<const double2*>(ap + g);
                    if (((k + 1) & (wch - 1)) == 0) E = eb[(k + 1) >> wlog];
                }
                r = *reinterpret_cast<const double2*>(wr + g);
                im = *reinterpret_cast<const double2*>(wi + g);
            }
            uint32_t q0[F64_SL], q1[F64_SL];
            f64_digits(f64_fix(w0.x * ac.x, E1), f64_fix(w0.y * ac.y, E1), q0);
            f64_digits(f64_fix(w1.x * ac.x, E1), f64_fix(w1.y * ac.y, E1), q1);
            if (k >= F64_GSTAGES) {
                const int kp = k - F64_GSTAGES;
                ok = mbar_wait_warp(done0 + 8 * (kp % F64_DONE), (kp / F64_DONE) & 1, abort_flag, A.err, 36, A.wait_limit);
            }
            if (!ok) break;
            unsigned char* bt = gsm + s * F64_GSTAGE;
#pragma unroll
            for (int i = 0; i < F64_SL; ++i) {
                *reinterpret_cast<uint32_t*>(bt + i * F64_B_TILE + ro) = q0[i];
                *reinterpret_cast<uint32_t*>(bt + i * F64_B_TILE + io) = q1[i];
            }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(gfull0 + 8 * s);
        }
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(F64_TMEM_COLS));
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
void f64_layout(const wpccc_basis_s* B, size_t node_doubles, ElemScratch& L) {
    auto a256 = [](size_t x) { return (x + 255) / 256 * 256; };
    L.tc_rows = 2 * B->N_T;
    L.Gp = (B->G + F64_K - 1) / F64_K * F64_K;
    L.f64_nwin = L.Gp / F64_K;
    size_t o = a256(node_doubles * sizeof(double));
    L.f64_pl = o;
    o += a256((size_t)F64_SL * L.tc_rows * L.Gp * 2);
    L.f64_ea = o;
    o += a256((size_t)L.f64_nwin * L.tc_rows * sizeof(int));
    L.f64_eb = o;
    o += a256((size_t)B->n_half * (B->dmax + 1) * L.f64_nwin * sizeof(int));
    L.f64_ap = o;
    o += a256((size_t)B->n_half * L.Gp * sizeof(double));
    L.f64_w2 = o;
    o += a256((size_t)2 * (B->dmax + 1) * L.Gp * sizeof(double));
    L.f64_r = o;
    o += a256((size_t)2 * L.Gp * sizeof(double));
    L.node_doubles = o / sizeof(double);
}

double f64_kappa(const wpccc_basis_s* B) { return std::min(std::fabs(B->T.Z), std::fabs(B->P.Z)); }

// Work lists of k_f64_slices, kept on the basis: (radial, |m|) items of the target and the half columns.
static wpccc_status f64_lists(wpccc_basis_s* B) {
    if (B->f64_items) return WPCCC_OK;
    std::vector<int> trow(2 * (size_t)B->N_T), hs(B->n_half);
    WPCCC_CUDA(cudaMemcpy(trow.data(), B->tc_row, trow.size() * sizeof(int), cudaMemcpyDeviceToHost));
    WPCCC_CUDA(cudaMemcpy(hs.data(), B->half_state, hs.size() * sizeof(int), cudaMemcpyDeviceToHost));
    std::vector<int> list, index((size_t)B->T.n_rad * (2 * WPCCC_LMAX + 1), -1);
    for (int i = 0; i < B->N_T; ++i) index[(size_t)B->T.h_st_rad[i] * (2 * WPCCC_LMAX + 1) + B->T.h_st_m[i] + WPCCC_LMAX] = i;
    int n = 0;
    for (int i = 0; i < B->N_T; ++i) {
        const int a = B->T.h_st_rad[i], l = B->T.h_rad_l[a], m = B->T.h_st_m[i];
        if (m < 0) continue;
        const int in = m > 0 ? index[(size_t)a * (2 * WPCCC_LMAX + 1) - m + WPCCC_LMAX] : -1;
        list.insert(list.end(), {a, l * (l + 1) / 2 + m, m & 1, trow[i], in >= 0 ? trow[in] : -1, trow[B->N_T + i],
                                 in >= 0 ? trow[B->N_T + in] : 0});
        ++n;
    }
    const size_t head = list.size();
    for (int c = 0; c < B->n_half; ++c) {
        const int a = B->P.h_st_rad[hs[c]], l = B->P.h_rad_l[a], q = B->P.h_st_m[hs[c]];
        list.insert(list.end(), {a, l * (l + 1) / 2 + q, q});
    }
    int* d = nullptr;
    WPCCC_CUDA(cudaMalloc((void**)&d, list.size() * sizeof(int)));
    cudaError_t e = cudaMemcpy(d, list.data(), list.size() * sizeof(int), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(d);
        return cuda_fail(e, "FP64 tensor-core contraction: work lists");
    }
    B->f64_items = d;
    B->f64_halves = d + head;
    B->n_f64_items = n;
    return WPCCC_OK;
}

wpccc_status fp64_route(wpccc_basis_s* B, int* precision) {
    *precision = ELEM_F64;
    if (B->n_centres != 2 || !encode_fn()) return WPCCC_OK;
    wpccc_status s = tc_prepare(B, false);
    if (s != WPCCC_OK) return s;
    if ((s = f64_lists(B)) != WPCCC_OK) return s;
    *precision = ELEM_F64_TC;
    return WPCCC_OK;
}

wpccc_status launch_mol_f64tc(wpccc_basis_s* B, const EvalDesc* evals, int nev, void* node, double2* mol, int* err,
                              cudaStream_t st) {
    const ElemScratch L = elem_scratch_layout(B, ELEM_F64_TC);
    const size_t node_bytes = L.node_doubles * sizeof(double);
    F64SliceArgs sa;
    sa.ev = evals;
    sa.kappa = f64_kappa(B);
    sa.G = B->G;
    sa.Gp = L.Gp;
    sa.nradT = B->T.n_rad;
    sa.nradP = B->P.n_rad;
    sa.nlqT = B->nlq_T;
    sa.nd = B->dmax + 1;
    sa.n_half = B->n_half;
    sa.tc_rows = L.tc_rows;
    sa.nwin = L.f64_nwin;
    sa.n_items = B->n_f64_items;
    sa.qmaxT = B->T.lmax;
    sa.items = B->f64_items;
    sa.halves = B->f64_halves;
    sa.node = static_cast<char*>(node);
    sa.node_bytes = node_bytes;
    sa.pl_off = L.f64_pl;
    sa.ea_off = L.f64_ea;
    sa.eb_off = L.f64_eb;
    sa.ap_off = L.f64_ap;
    sa.w2_off = L.f64_w2;
    sa.r_off = L.f64_r;
    const size_t ssm = (size_t)sa.nd * F64_WIN * sizeof(int);
    if (ssm > 40 * 1024)   // with the static 8 KB
        WPCCC_CUDA(cudaFuncSetAttribute(k_f64_slices, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssm));
    k_f64_slices<<<dim3((sa.Gp + F64_WIN - 1) / F64_WIN * F64_SPLIT, nev), 256, ssm, st>>>(sa);
    WPCCC_CHECK_LAUNCH("k_f64_slices");
    // the digit planes as one 3-D bf16 tensor: x = node (Gp), y = digit plane row (8 x tc_rows), z = position
    F64Maps maps;
    const cuuint64_t dims[3] = {(cuuint64_t)L.Gp, (cuuint64_t)F64_SL * L.tc_rows, (cuuint64_t)nev};
    const cuuint64_t strides[2] = {(cuuint64_t)L.Gp * 2, (cuuint64_t)node_bytes};
    const cuuint32_t estr[3] = {1, 1, 1};
    for (int h = 0; h < F64_M / 32; ++h) {
        const cuuint32_t bx[3] = {(cuuint32_t)F64_K, (cuuint32_t)(32 * (h + 1)), 1};
        CUresult r = encode_fn()(&maps.m[h], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, static_cast<char*>(node) + L.f64_pl, dims,
                                 strides, bx, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return fail(WPCCC_ECUDA, "cuTensorMapEncodeTiled failed for the digit planes");
    }
    F64Args a;
    a.ev = evals;
    a.kappa = f64_kappa(B);
    a.Gp = L.Gp;
    a.N_T = B->N_T;
    a.n_half = B->n_half;
    a.nk = L.Gp / F64_K;
    a.nwin = L.f64_nwin;
    a.nd = B->dmax + 1;
    a.n_ntiles = (B->n_half + F64_HALF - 1) / F64_HALF;
    a.tc_rows = L.tc_rows;
    a.qg_max = B->qg_max;
    a.qg_off = B->qg_off;
    a.qg_q = B->qg_off + B->n_qgroups + 1;
    a.qg_rows = B->qg_rows;
    a.half_q = B->tc_halfq;
    a.node = static_cast<const char*>(node);
    a.node_bytes = node_bytes;
    a.ea_off = L.f64_ea;
    a.eb_off = L.f64_eb;
    a.ap_off = L.f64_ap;
    a.w2_off = L.f64_w2;
    a.mol = reinterpret_cast<double*>(mol);
    a.err = err;
    a.wait_limit = B->wait_polls;
    const size_t smem = 1024 + F64_RING + (size_t)F64_GSTAGES * F64_GSTAGE;
    WPCCC_CUDA(cudaFuncSetAttribute(k_mol_f64tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_mol_f64tc<<<dim3(a.n_ntiles * B->n_qgroups, nev), F64_THREADS, smem, st>>>(maps, a);
    WPCCC_CHECK_LAUNCH("k_mol_f64tc");
    return WPCCC_OK;
}

}  // namespace wpccc
