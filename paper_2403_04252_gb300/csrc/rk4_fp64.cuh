// The FP64 forms' RK4 sweep (Algorithm 1): one cluster of one to eight blocks per path.
//
//   RK_MATRIX  X = S^{-1} H stored (the paper's form; one-centre: X = H)
//   RK_STAGE   S^{-1} applied from FP64 LU factors at every stage
//   RK_SCHUR   S^{-1} applied through the Schur complement's Cholesky factor at every stage
//
// What bounds it: a stage multiplies the path's vector by matrices that are read once, at two FP64 multiply-adds per clock
// per SM (N = 59: 3.4 us of FP64 pipe per stage on one SM; N = 380, Schur form: 250 us), after load latencies and
// barriers that one row per thread leaves uncovered.  So the rows of every product are shared out over the cluster, and
// within a block over groups of threads that take the columns in turn; the input vector is replicated in every block's
// shared memory, and the thread that finishes a row stores it into all of them (distributed shared memory).  Two
// copies of the input vector take turns, so that one cluster barrier per stage suffices.  The triangular solves go
// panel by panel (32 rows, the panels to the blocks in turn): the owner solves the diagonal block and sends the 32
// unknowns to all blocks, every block updates its own rows; the factor's tile is loaded before the barrier.
// Measured, one block per path with a row per thread -> here, sweeps alone: one centre, N = 59, 8 paths of 800 steps
// 42.6 -> 10.2 ms (13.3 -> 3.2 us per stage); two centres, LU, N = 109, 5 paths of 11 to 23 steps 10.3 -> 4.4 ms (inverted
// diagonal blocks included, see rc_lu_solve); Schur, N = 380, 32 paths of 10 steps 22 -> 9.0 ms.  Slopes are formed with
// 1 / v, one rounding more than a division by v.
#pragma once

#include "cluster.cuh"
#include "rk_device.cuh"

namespace wpccc {

constexpr int RC_THREADS = 512;
constexpr int RC_BLK = RC_THREADS;   // double2 of block scratch: partial sums, or pivots

static __device__ __forceinline__ void remote_store(uint32_t addr, int rank, double2 v) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};\n" ::"r"(r), "d"(v.x), "d"(v.y) : "memory");
}

struct RcCluster {
    int rank, size;
    // v into *p of every block's shared memory
    __device__ __forceinline__ void bcast(double2* p, double2 v) const {
        if (size == 1) {
            *p = v;
            return;
        }
        const uint32_t a = smem_u32(p);
        for (int r = 0; r < size; ++r) remote_store(a, r, v);
    }
    __device__ __forceinline__ void sync() const {
        if (size == 1) __syncthreads();
        else cluster_sync_all();
    }
    // rows [lo, hi) of n for this block: contiguous, in multiples of eight (128 bytes of a column)
    __device__ __forceinline__ void rows(int n, int& lo, int& hi) const {
        const int per = ((n + size - 1) / size + 7) / 8 * 8;
        lo = min(n, rank * per);
        hi = min(n, lo + per);
    }
};

// Sums of the groups' partial results, in order: part[g rb + slot] for g < RC_G.  A thread per real and imaginary part
// (an FP64 instruction holds its quarter's pipe for 64 cycles, so the chain is halved); epi(row, value) runs on the
// even threads.
constexpr int RC_G = 8;
template <typename F>
static __device__ __forceinline__ void rc_reduce(const double2* part, int rb, int base, int nr, F epi) {
    const int tid = threadIdx.x;
    if (tid < ((2 * rb + 31) & ~31)) {   // whole warps
        const int slot = min(tid >> 1, rb - 1);
        const double* p = reinterpret_cast<const double*>(part + slot) + (tid & 1);
        double a = p[0];
#pragma unroll
        for (int g = 1; g < RC_G; ++g) a += p[2 * g * rb];
        const double b = __shfl_down_sync(0xffffffffu, a, 1);
        if ((tid & 1) == 0 && tid < 2 * rb && base + slot < nr) epi(base + slot, make_double2(a, b));
    }
}

// (M x)_row for nr rows from M (column-major, leading dimension ld, nc columns), handed to epi(row, value) by one thread
// per row.  Eight groups of threads take the columns in turn, up to 64 rows per pass; their partial sums meet in
// `part` (RC_THREADS entries) and are added in order, so a result does not depend on the cluster's size.  load() brings
// the first entries of a thread's share into registers ahead of the vector; keep the object to use them again.
struct RcRows {
    static constexpr int PRE = 8;
    double2 a[PRE];
    __device__ __forceinline__ void load(const double2* __restrict__ M, size_t ld, int nr, int nc) {
        const int rb = min(RC_THREADS / RC_G, (nr + 7) & ~7), tid = threadIdx.x;
        const int slot = rb ? tid % rb : 0, grp = rb ? tid / rb : RC_G;
#pragma unroll
        for (int q = 0; q < PRE; ++q) {
            const int j = grp + q * RC_G;
            a[q] = (grp < RC_G && slot < nr && j < nc) ? M[slot + (size_t)j * ld] : make_double2(0.0, 0.0);
        }
    }
    template <typename F>
    __device__ __forceinline__ void apply(const double2* __restrict__ M, size_t ld, int nr, int nc, const double2* x,
                                          double2* part, F epi) const {
        if (nr <= 0) return;
        const int tid = threadIdx.x;
        const int rb = min(RC_THREADS / RC_G, (nr + 7) & ~7);
        const int slot = tid % rb, grp = tid / rb;
        for (int base = 0; base < nr; base += rb) {
            const int row = base + slot;
            if (grp < RC_G) {
                double re = 0.0, im = 0.0;
                auto step = [&](double2 m, double2 q) {
                    re = fma(m.x, q.x, re);
                    re = fma(-m.y, q.y, re);
                    im = fma(m.x, q.y, im);
                    im = fma(m.y, q.x, im);
                };
                int j = grp;
                if (base == 0) {
#pragma unroll
                    for (int q = 0; q < PRE; ++q, j += RC_G)
                        if (j < nc) step(a[q], x[j]);
                }
                if (row < nr) {
                    const double2* p = M + row + (size_t)j * ld;
                    const size_t inc = (size_t)RC_G * ld;
#pragma unroll 8
                    for (; j < nc; j += RC_G, p += inc) step(*p, x[j]);
                }
                part[tid] = make_double2(re, im);
            }
            __syncthreads();
            rc_reduce(part, rb, base, nr, epi);
            __syncthreads();
        }
    }
};
template <typename F>
static __device__ __forceinline__ void rc_matvec(const double2* __restrict__ M, size_t ld, int nr, int nc,
                                                 const double2* x, double2* part, F epi) {
    RcRows R;
    R.load(M, ld, nr, nc);
    R.apply(M, ld, nr, nc, x, part, epi);
}

// One panel's update of this block's own rows: w[r] -= sum_{j < nb} M[r][j] x[j] for the rows of its panels q0, q0 + size,
// ... (cnt panels of 32 rows, n rows in all), M at the panel's first column.  Four groups of threads take the columns
// in turn, up to four panels per pass; the first pass's entries are loaded by load(), before the barrier that makes x
// known.
struct RcPanel {
    static constexpr int G = 4, PER = 32 / G;
    double2 a[PER];
    int rb, slot, grp, cnt, q0, size, n;
    const double2* M;
    size_t ld;
    __device__ __forceinline__ int row_of(int s) const { return (q0 + (s >> 5) * size) * 32 + (s & 31); }
    __device__ __forceinline__ void fetch(int s, int nb) {
        const int r = row_of(s);
        const bool on = grp < G && s < cnt * 32 && r < n;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int j = grp + q * G;
            a[q] = (on && j < nb) ? M[(size_t)r + (size_t)j * ld] : make_double2(0.0, 0.0);
        }
    }
    __device__ __forceinline__ void load(const double2* M_, size_t ld_, int q0_, int cnt_, int size_, int n_, int nb) {
        M = M_;
        ld = ld_;
        q0 = q0_;
        cnt = cnt_;
        size = size_;
        n = n_;
        if (cnt <= 0) return;
        rb = min(RC_THREADS / G, cnt * 32);
        slot = (int)threadIdx.x % rb;
        grp = (int)threadIdx.x / rb;
        fetch(slot, nb);
    }
    __device__ __forceinline__ void apply(const double2* x, double2* w, int nb, double2* part) {
        for (int base = 0; base < cnt * 32; base += rb) {
            if (base > 0) fetch(base + slot, nb);
            const int r = row_of(base + slot);
            double re = 0.0, im = 0.0;
            if (grp < G) {
#pragma unroll
                for (int q = 0; q < PER; ++q) {
                    const int j = grp + q * G;
                    const double2 v = x[j < nb ? j : 0];   // the entries past nb are zero
                    re = fma(a[q].x, v.x, re);
                    re = fma(-a[q].y, v.y, re);
                    im = fma(a[q].x, v.y, im);
                    im = fma(a[q].y, v.x, im);
                }
                part[threadIdx.x] = make_double2(re, im);
            }
            __syncthreads();
            if (grp == 0 && base + slot < cnt * 32 && r < n) {
#pragma unroll
                for (int g = 1; g < G; ++g) {
                    const double2 o = part[g * rb + slot];
                    re += o.x;
                    im += o.y;
                }
                w[r] = make_double2(w[r].x - re, w[r].y - im);
            }
            __syncthreads();
        }
    }
};

// First own panel after p (or the number of own panels before p), for panels q with q % size == rank.
static __device__ __forceinline__ int rc_first_after(int p, int rank, int size) {
    const int q = p + 1;
    return q + (rank - q % size + size) % size;
}
static __device__ __forceinline__ int rc_count(int first, int end, int size) {
    return first < end ? (end - first + size - 1) / size : 0;
}

// S = [[I, K], [K^+, I]]: t <- S^{-1} t (replicated in every block, N entries), with L's panels as k_schur_factor<double>
// leaves them: L below the diagonal blocks, L^+ above them, L_pp^{-1} in the lower and its adjoint in the upper half
// of the diagonal blocks.  z: scratch of N - N_T entries (replicated).  On return t holds x_P in its projectile part
// everywhere, the target part is left to the caller's last product (t_T - K x_P).
static __device__ __noinline__ void rc_schur_solve(const RcCluster& cl, const double2* __restrict__ S, int N, int N_T,
                                                      double2* t, double2* z, double2* part) {
    const int NP = N - N_T, np = (NP + 31) / 32;
    const double2* C = S + N_T + (size_t)N_T * N;
    double2* tp = t + N_T;
    // u_P = t_P - K^+ t_T
    int lo, hi;
    cl.rows(NP, lo, hi);
    rc_matvec(S + N_T + lo, N, hi - lo, N_T, t, part, [&](int r, double2 v) {
        cl.bcast(z + lo + r, make_double2(tp[lo + r].x - v.x, tp[lo + r].y - v.y));
    });
    cl.sync();
    RcPanel P;
    const int tid = threadIdx.x;
    // diagonal block p times w (lower = its inverse, upper = the inverse's adjoint): 16 threads per row
    auto diag = [&](int p, const double2* w, bool upper, double2* out) {
        const int nb = min(32, NP - 32 * p), r = tid >> 4, l = tid & 15;
        double re = 0.0, im = 0.0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = l + 16 * h;
            if (r < nb && j < nb && (upper ? j >= r : j <= r)) {
                const double2 m = C[(size_t)(32 * p + r) + (size_t)(32 * p + j) * N];
                const double2 v = w[32 * p + j];
                re += m.x * v.x - m.y * v.y;
                im += m.x * v.y + m.y * v.x;
            }
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            re += __shfl_xor_sync(0xffffffffu, re, o);
            im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        if (l == 0 && r < nb) cl.bcast(out + 32 * p + r, make_double2(re, im));
    };
    // L z = u: z holds the right-hand side (own panels) and receives no results: they go to t_P
    for (int p = 0; p < np; ++p) {
        if (p % cl.size == cl.rank) diag(p, z, false, tp);
        const int q0 = rc_first_after(p, cl.rank, cl.size);
        P.load(C + (size_t)(32 * p) * N, N, q0, rc_count(q0, np, cl.size), cl.size, NP, min(32, NP - 32 * p));
        cl.sync();
        P.apply(tp + 32 * p, z, min(32, NP - 32 * p), part);
        __syncthreads();
    }
    // L^+ x = z: own panels of the right-hand side back from t_P
    for (int r = tid; r < NP; r += RC_THREADS)
        if ((r >> 5) % cl.size == cl.rank) z[r] = tp[r];
    __syncthreads();
    for (int p = np - 1; p >= 0; --p) {
        if (p % cl.size == cl.rank) diag(p, z, true, tp);
        P.load(C + (size_t)(32 * p) * N, N, cl.rank, rc_count(cl.rank, p, cl.size), cl.size, NP, min(32, NP - 32 * p));
        cl.sync();
        P.apply(tp + 32 * p, z, min(32, NP - 32 * p), part);
        __syncthreads();
    }
}

// t <- S^{-1} t (replicated) from P S = L U with inverted 32 x 32 diagonal blocks (launch_lu_invert_diag): perm[r] = row of t
// that comes r-th.  z: scratch of N entries; part: RC_BLK.  The inverse turns a panel's chain of 32 dependent FP64 steps
// into one product of 16 threads per row, whose entries are loaded before the barrier that makes the panel's right-hand
// side known (N = 109, 5 paths of 11 to 23 steps: sweep 7.8 -> 4.4 ms, for 0.3 ms of inversion; the adjoint of p + Li,
// N = 379: 35 -> 28 ms).
static __device__ __noinline__ void rc_lu_solve(const RcCluster& cl, const double2* __restrict__ LU, const uint16_t* perm,
                                                   int N, double2* t, double2* z, double2* part) {
    const int np = (N + 31) / 32, tid = threadIdx.x, dr = tid >> 4, dl = tid & 15;
    double2 m[2];   // this thread's entries (dr, dl) and (dr, dl + 16) of the next own diagonal block
    auto fetch = [&](int p, bool upper) {
        if (p < 0 || p >= np || p % cl.size != cl.rank) return;
        const int nb = min(32, N - 32 * p);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = dl + 16 * h;
            m[h] = make_double2(!upper && j == dr ? 1.0 : 0.0, 0.0);
            if (dr < nb && j < nb && (upper ? j >= dr : j < dr)) m[h] = LU[(size_t)(32 * p + dr) + (size_t)(32 * p + j) * N];
        }
    };
    auto diag = [&](int p) {
        if (p % cl.size != cl.rank) return;
        const int nb = min(32, N - 32 * p);
        double re = 0.0, im = 0.0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = dl + 16 * h;
            const double2 v = z[32 * p + (j < nb ? j : 0)];   // the entries past nb are zero
            if (j < nb) {
                re += m[h].x * v.x - m[h].y * v.y;
                im += m[h].x * v.y + m[h].y * v.x;
            }
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            re += __shfl_xor_sync(0xffffffffu, re, o);
            im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        if (dl == 0 && dr < nb) cl.bcast(t + 32 * p + dr, make_double2(re, im));
    };
    fetch(0, false);
    for (int r = tid; r < N; r += RC_THREADS)
        if ((r >> 5) % cl.size == cl.rank) z[r] = t[perm[r]];
    cl.sync();   // t may be overwritten
    RcPanel P;
    for (int p = 0; p < np; ++p) {
        const int nb = min(32, N - 32 * p);
        diag(p);
        fetch(p + 1, false);
        const int q0 = rc_first_after(p, cl.rank, cl.size);
        P.load(LU + (size_t)(32 * p) * N, N, q0, rc_count(q0, np, cl.size), cl.size, N, nb);
        cl.sync();
        P.apply(t + 32 * p, z, nb, part);
        __syncthreads();
    }
    fetch(np - 1, true);
    for (int r = tid; r < N; r += RC_THREADS)
        if ((r >> 5) % cl.size == cl.rank) z[r] = t[r];
    __syncthreads();
    for (int p = np - 1; p >= 0; --p) {
        const int nb = min(32, N - 32 * p);
        diag(p);
        fetch(p - 1, true);
        P.load(LU + (size_t)(32 * p) * N, N, cl.rank, rc_count(cl.rank, p, cl.size), cl.size, N, nb);
        cl.sync();
        P.apply(t + 32 * p, z, nb, part);
        __syncthreads();
    }
}

// Row order of LAPACK pivots (1-based): perm[r] = the row that the interchanges bring to r.
static __device__ __forceinline__ void rc_permutation(const int* __restrict__ piv, int N, uint16_t* perm, double2* scratch) {
    int* s = reinterpret_cast<int*>(scratch);   // RC_BLK double2: the pivots, 2048 at a time
    for (int r = threadIdx.x; r < N; r += RC_THREADS) perm[r] = (uint16_t)r;
    for (int b = 0; b < N; b += 2048) {
        const int n = min(2048, N - b);
        __syncthreads();
        for (int r = threadIdx.x; r < n; r += RC_THREADS) s[r] = piv[b + r] - 1;
        __syncthreads();
        if (threadIdx.x == 0)
            for (int r = 0; r < n; ++r) {
                const int p = s[r];
                if (p != b + r) {
                    const uint16_t q = perm[b + r];
                    perm[b + r] = perm[p];
                    perm[p] = q;
                }
            }
    }
    __syncthreads();
}

// Blocks per path of the cluster sweeps: as many as `share` SMs allow, with at least eight rows of the vector each.  The
// results do not depend on it.
static inline int rk4_cluster(int npc, int N, int share) {
    int cl = 1;
    while (cl < 8 && 2 * cl * npc <= share && N >= 14 * cl) cl *= 2;
    return cl;
}

}  // namespace wpccc
