// csrc/f64_order.cuh on the host.  Arguments: Geta, Gtau, kappa R, then any number of tau.  Prints the window length in
// nodes, the original index of every node in order, and the scale exponent at each tau, a line each.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>

using std::fmin;
using std::max;
using std::min;
static double __dmul_rn(double a, double b) { return a * b; }
static double __ddiv_rn(double a, double b) { return a / b; }
static int __double2int_rn(double x) { return (int)std::nearbyint(x); }
#define __device__
#define __forceinline__ inline
#include "f64_order.cuh"

int main(int argc, char** argv) {
    const int Ge = std::atoi(argv[1]), Gt = std::atoi(argv[2]);
    const double kR = std::atof(argv[3]);
    std::printf("%d\n", 32 * wpccc::f64_window_chunks((Ge * Gt + 31) / 32 * 32, kR));
    const int width = wpccc::f64_block_width(Ge, Gt, kR);
    for (int g = 0; g < Ge * Gt; ++g) {
        int k, t;
        wpccc::f64_node(g, Ge, Gt, width, k, t);
        std::printf("%d ", k * Gt + t);
    }
    std::printf("\n");
    for (int i = 4; i < argc; ++i) std::printf("%d ", wpccc::f64_scale(kR, std::atof(argv[i])));
    std::printf("\n");
}
