// csrc/chol_panel.cuh on the host: one host thread per GPU thread, barriers for __syncthreads and __syncwarp, and every
// access to the block's shared arrays recorded.  Two accesses of different threads to one word, one of them a store, must
// have a block barrier between them, or a warp barrier when the threads share a warp.  Prints the number of pairs of
// accesses without one and the largest error of L L^+ against the block.
#include <barrier>
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <memory>
#include <random>
#include <thread>
#include <vector>

constexpr int WARPS = 8, THREADS = 32 * WARPS, LD = 33;
struct Access { const void* at; bool store; int block, warp; };
static thread_local int me = 0, block_epoch = 0, warp_epoch = 0;
static std::vector<Access> trace[THREADS];
static const char *lo[2], *hi[2];
static void note(const void* p, bool store) {
    const char* q = static_cast<const char*>(p);
    if ((q >= lo[0] && q < hi[0]) || (q >= lo[1] && q < hi[1])) trace[me].push_back({p, store, block_epoch, warp_epoch});
}
struct Real {
    double v;
    Real(double x = 0) : v(x) {}
    Real(const Real& o) : v(o) {}
    Real& operator=(const Real& o) { const double x = o; note(this, true); v = x; return *this; }
    Real& operator-=(double x) { return *this = Real(double(*this) - x); }
    operator double() const { note(this, false); return v; }
};
struct double2 { Real x, y; };
struct float2 { float x, y; };
static double2 make_double2(double x, double y) { return {x, y}; }
static float2 make_float2(float x, float y) { return {x, y}; }
static float rsqrtf(float x) { return 1.f / std::sqrt(x); }
static double rsqrt(double x) { return 1.0 / std::sqrt(x); }

static std::unique_ptr<std::barrier<>> all, some[WARPS];
static void __syncthreads() { all->arrive_and_wait(); ++block_epoch; ++warp_epoch; }
static void __syncwarp() { some[me / 32]->arrive_and_wait(); ++warp_epoch; }
#define __device__
#define __forceinline__ inline
using std::fma;
using std::sqrt;
#include "chol_panel.cuh"

int main(int argc, char** argv) {
    const int nb = argc > 1 ? std::atoi(argv[1]) : 32;
    static double2 sL[32 * LD];
    static Real s_inv[32];
    int info = 0;
    lo[0] = reinterpret_cast<char*>(sL), hi[0] = lo[0] + sizeof sL;
    lo[1] = reinterpret_cast<char*>(s_inv), hi[1] = lo[1] + sizeof s_inv;
    std::mt19937 gen(7);
    std::normal_distribution<double> n;
    using Z = std::complex<double>;
    std::vector<Z> K(nb * nb), C(nb * nb);
    for (auto& k : K) k = Z(n(gen), n(gen)) * 0.1;
    for (int i = 0; i < nb; ++i)
        for (int j = 0; j <= i; ++j) {
            Z s = i == j ? 1.0 : 0.0;
            for (int k = 0; k < nb; ++k) s += K[i * nb + k] * std::conj(K[j * nb + k]);
            C[i * nb + j] = s;
            sL[j * LD + i].x.v = s.real();
            sL[j * LD + i].y.v = s.imag();
        }
    all = std::make_unique<std::barrier<>>(THREADS);
    for (auto& b : some) b = std::make_unique<std::barrier<>>(32);
    std::vector<std::thread> t;
    for (int i = 0; i < THREADS; ++i)
        t.emplace_back([&, i] {
            me = i;
            wpccc::chol_diag_block<WARPS>(sL, LD, s_inv, &info, 0, nb, i);
        });
    for (auto& x : t) x.join();
    std::map<const void*, std::vector<std::pair<int, const Access*>>> by;
    for (int i = 0; i < THREADS; ++i)
        for (const Access& a : trace[i]) by[a.at].push_back({i, &a});
    long open = 0;
    for (auto& [at, v] : by)
        for (auto& [ti, a] : v)
            for (auto& [tj, b] : v) {
                if (!a->store || ti == tj || a->block != b->block) continue;
                if (ti / 32 == tj / 32 && a->warp != b->warp) continue;
                if (!b->store || ti < tj) ++open;
            }
    double err = 0.0;
    for (int i = 0; i < nb; ++i)
        for (int j = 0; j <= i; ++j) {
            Z s = 0.0;
            for (int k = 0; k <= j; ++k)
                s += Z(sL[k * LD + i].x.v, sL[k * LD + i].y.v) * std::conj(Z(sL[k * LD + j].x.v, sL[k * LD + j].y.v));
            err = std::max(err, std::abs(s - C[i * nb + j]));
        }
    std::printf("%ld %.3e %d\n", open, err, info);
}
