// Order of the quadrature nodes, length of the scaling windows and power-of-two scales of the FP64 contraction in digits
// (mol_fp64.cu).  tests/test_f64_order.py compiles this file for the host.
//
// A window's digits are fixed point against the product of two maxima, so a sum keeps FP64's relative accuracy only where
// both operand rows are large at the same nodes of the window.  A target row falls like exp(-kappa r_T), a projectile row
// like exp(-kappa r_P) (kappa: the smaller charge, the steepest slope both have), r_T, r_P = (R / 2)(eta +- tau): along eta
// they fall together, along tau against each other.  Three measures, all exact or free:
//   - nodes in blocks of neighbouring tau, within a block by eta, so that a window spans a short stretch of both;
//   - windows of 512 terms near the target, 128, 64 or 32 further out: the more the larger kappa R;
//   - row A times 2^s, row B times 2^-s with 2^s near exp((kappa R / 4) tau), which halves the slopes of the steep rows.
// Error of an element by rounding the operands, in units of 2^-53 sum |terms| (largest over the elements, and median), for
// windows of 512 nodes over all tau -> here -> a chain of FP64 multiply-adds; p + H, N = 380, b = 1:
//   z =  8: 12, 0.04 -> 1.5, 0.04 -> 30, 0.7      z = 30: 4e9, 0.1 -> 1.2, 0.07 -> 15, 0.4
//   z = 16: 2e3, 0.06 -> 2.2, 0.05 -> 21, 0.4     z = 40: 3e13, 0.2 -> 2.3, 0.2 -> 26, 0.3
//   z = 24: 3e6, 0.09 -> 15, 0.09 -> 21, 0.3      z = 80: 6e14, 0.3 -> 1.1, 0.1 -> 20, 0.3
// and as well at or below the chain's for C6+ + H, He+ + He+ and rules of 24 x 16 to 128 x 48 nodes at these kappa R.  Where it
// ends: p + H stays below 40 up to kappa R = 150 and reaches 90 at 180, charges of 6 on both centres reach 100 from 144 on,
// and rules too coarse for the distance 200 (31 x 7 nodes at kappa R = 40, 16 x 16 at 50).
#pragma once

namespace wpccc {

// tau nodes per block: a sixth of them, fewer from kappa R = 48 on; one more where a block of few eta nodes then ends on a
// window's boundary (24 x 16 nodes, kappa R = 40: 1400 units with three, 9 with four).
static __device__ __forceinline__ int f64_block_width(int Geta, int Gtau, double kR) {
    const int w = max(1, min((Gtau + 3) / 6, (int)fmin(__ddiv_rn(8.0 * Gtau, kR), 1e6)));
    return Geta <= 32 && w * Geta % 32 != 0 && (w + 1) * Geta % 32 == 0 ? w + 1 : w;
}

// Node g of the order: eta index k, tau index t.
static __device__ __forceinline__ void f64_node(int g, int Geta, int Gtau, int width, int& k, int& t) {
    const int block = g / (width * Geta), rest = g - block * width * Geta, w = min(width, Gtau - block * width);
    k = rest / w;
    t = block * width + rest - k * w;
}

// Chunks of 32 terms per window: (kappa R)^2 / 48 windows of G terms, in lengths of 512, 128, 64 and 32 (256 gains nothing
// over 512 in accuracy).
static __device__ __forceinline__ int f64_window_chunks(int G, double kR) {
    const double q = __dmul_rn(kR, kR), lim = 48.0 * G;
    return 512.0 * q <= lim ? 16 : 128.0 * q <= lim ? 4 : 64.0 * q <= lim ? 2 : 1;
}

// Exponent s of the scale at tau: (kappa R / 4) tau log2(e), as far as FP64's range allows.
static __device__ __forceinline__ int f64_scale(double kR, double tau) {
    return __double2int_rn(0.25 * 1.4426950408889634 * fmin(kR, 400.0) * tau);
}

}  // namespace wpccc
