// Building blocks of the contractions that the tensor cores carry out in FP64's place (mol_fp64.cu,
// schur_fp64.cu): fixed-point digits of FP64 rows, the MMAs of one chunk, and the sums put together again.
// The representation and its error are described in mol_fp64.cu.
#pragma once

#include <cstdint>

#include "tc_ptx.cuh"

namespace wpccc {

constexpr int F64_SL = 8;                       // digits per operand
constexpr int F64_LEV = 9;                      // levels 0..8
constexpr int F64_M = 128;                      // A rows per CTA (MMA M)
constexpr int F64_N = 32;                       // B rows per CTA (MMA N of one digit)
constexpr int F64_K = 32;                       // terms per chunk: one 64-byte bf16 row
constexpr int F64_WIN = 512;                    // terms per scaling window, at most
constexpr int F64_WCH = F64_WIN / F64_K;        // chunks per window
constexpr int F64_TMEM_COLS = 512;              // one buffer of accumulators: 9 x 32 = 288 columns
constexpr int F64_B_TILE = F64_N * 64;          // bytes of one digit of the B tile
static_assert(F64_LEV * F64_N <= F64_TMEM_COLS && (F64_LEV - 1) * F64_N <= 256, "accumulators; widest MMA");
constexpr int F64_BAD = 1 << 14;                // scale exponent of a row with a non-finite value
constexpr int F64_EMIN = -900, F64_EMAX = 1000; // range of the scale exponents
// 64 in each of the eight seven-bit digits: a fixed-point number plus this has the balanced digits as bit fields.
constexpr uint64_t F64_BIAS = 64ull | 64ull << 7 | 64ull << 14 | 64ull << 21 | 64ull << 28 | 64ull << 35 | 64ull << 42 | 64ull << 49;

// x in fixed point against 2^E: X + F64_BIAS with X = x 2^(55 - E) rounded to nearest (|x| < 0.992 2^E, so
// |X| < 2^55); E1 = E + 1023.  Denormals read as zero (E >= F64_EMIN is far above them).
static __device__ __forceinline__ uint64_t f64_fix(double x, int E1) {
    const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
    const uint32_t s = min((uint32_t)(E1 - (int)((h >> 20) & 0x7FFu)), 63u);
    const uint64_t m = ((uint64_t)(((h & 0xFFFFFu) | 0x100000u) << 4 | l >> 28) << 32) | (uint64_t)(l << 4);
    const uint64_t q = ((m >> s) + 1) >> 1, sm = (uint64_t)(int64_t)((int32_t)h >> 31);
    return F64_BIAS + ((q ^ sm) - sm);
}

// Scale exponent E of a row from the largest sign-stripped high word: |x| < 0.992 2^E (the digits' range is
// (1 - 1/127) 2^51, so the mantissa is taken 1 % larger).
static __device__ __forceinline__ int f64_exponent(int hmax, int margin) {
    if (hmax >= 0x7FF00000) return F64_BAD;
    const int E = ((hmax + margin) >> 20) - 1022;
    return E > F64_EMAX ? F64_BAD : max(E, F64_EMIN);
}
constexpr int F64_MARGIN = 20000;               // 0.95 % of a mantissa unit, above 1/127 of half of it
// the sum of two high words under-estimates the logarithm of a product by up to 0.172 (piecewise linear log2)
constexpr int F64_MARGIN2 = 201000;

// Digit i of two values as bf16x2 numbers k 2^(-7 i), k in [-64, 63]: the digits plus 64 in the low seven bits of a
// and b become (128 + digit) 2^(-7 i) by their bit pattern, then 192 2^(-7 i) is subtracted (exact).
static __device__ __forceinline__ uint32_t f64_pair(uint32_t a, uint32_t b, int i) {
    const uint32_t sc = (uint32_t)(7 * i) * 0x00800080u;   // the exponents lowered by 7 i
    const uint32_t z = (__byte_perm(a, b, 0x5410) & 0x007F007Fu) | (0x43004300u - sc), c = 0x43404340u - sc;
    const __nv_bfloat162 v =
        __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&z), *reinterpret_cast<const __nv_bfloat162*>(&c));
    return *reinterpret_cast<const uint32_t*>(&v);
}

// The eight digits of two fixed-point values, packed as bf16x2.
static __device__ __forceinline__ void f64_digits(uint64_t x, uint64_t y, uint32_t out[F64_SL]) {
    const uint32_t xh = (uint32_t)(x >> 32), xl = (uint32_t)x, yh = (uint32_t)(y >> 32), yl = (uint32_t)y;
    out[0] = f64_pair(xh >> 17, yh >> 17, 0);
    out[1] = f64_pair(xh >> 10, yh >> 10, 1);
    out[2] = f64_pair(xh >> 3, yh >> 3, 2);
    out[3] = f64_pair(__funnelshift_r(xl, xh, 28), __funnelshift_r(yl, yh, 28), 3);
    out[4] = f64_pair(xl >> 21, yl >> 21, 4);
    out[5] = f64_pair(xl >> 14, yl >> 14, 5);
    out[6] = f64_pair(xl >> 7, yl >> 7, 6);
    out[7] = f64_pair(xl, yl, 7);
}

static __device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7FFFFFFF; }

// The nine levels of one element put together: 2^28 hi + lo in units of level 7 (2^(E - 61)), its top bits as one 51-bit
// integer T (units 2^(E - 42)), the low 19 apart.  Level 8 is rounded to level 7's unit.
static __device__ __forceinline__ void f64_levels(const float (&v)[F64_LEV][4], int u, long long& T, uint32_t& low19) {
    int L[F64_SL];
#pragma unroll
    for (int q = 0; q < F64_SL - 1; ++q) L[q] = __float2int_rn(v[q][u] * (float)(1ull << (7 * q)));
    L[7] = __float2int_rn((v[7][u] + v[8][u]) * (float)(1ull << 49));
    const long long hi = (long long)(L[0] * 128 + L[1]) * 16384 + (L[2] * 128 + L[3]);
    const long long lo = (long long)(L[4] * 128 + L[5]) * 16384 + (L[6] * 128 + L[7]);
    T = (hi << 9) + (lo >> 19);
    low19 = (uint32_t)lo & 0x7FFFFu;
}

// One window's sum added to the running sum: T 2^(E - 42) to acc (one FP64 FMA), the low part 2^(E - 61) to low in FP32, in
// units of 2^-unit, which keeps it for windows of 2^E from 2^(-65 - unit) to 2^(164 - unit) (-1000 < unit < 1000).  Zero
// below FP64's range, NaN for a row with a non-finite value.
constexpr int F64_UNIT = 100;
static __device__ __forceinline__ void f64_accumulate(double& acc, float& low, long long T, uint32_t low19, int E, int unit) {
    const double X = __dsub_rn(__longlong_as_double(T + 0x4338000000000000ll), 6755399441055744.0);
    const int es = E - 42 + 1023, ef = E - 61 + unit + 127;
    const int sh = E >= F64_BAD / 2 ? 0x7FF80000 : (max(0, min(es, 2046)) << 20);
    acc = fma(X, __hiloint2double(sh, 0), acc);
    const float r = __fsub_rn(__uint_as_float(0x4B000000u | low19), 8388608.f);
    low = fmaf(r, __uint_as_float((uint32_t)max(0, min(ef, 230)) << 23), low);
}
static __device__ __forceinline__ double f64_total(double acc, float low, int unit) {
    return fma((double)low, __hiloint2double((1023 - unit) << 20, 0), acc);
}

// The MMAs of one chunk (one thread): the B tile's digits lie one after the other, so one MMA per A digit and K step forms
// A_i [B_0 .. B_{8-i}] into the columns of levels i .. 8.  da, db: descriptors of the chunk's first digits, a16: bytes of
// an A digit / 16; fresh: the window's first products overwrite the accumulators.  between() runs while MMAs are queued: the
// queue is short, so what the issuing thread does between two chunks shows in full.
template <typename F>
static __device__ __forceinline__ void f64_mma_chunk(uint32_t tmem, uint64_t da, uint64_t db, uint32_t a16, bool fresh, F between) {
#pragma unroll
    for (int kk = 0; kk < F64_K / 16; ++kk) {
#pragma unroll
        for (int i = 0; i < F64_SL; ++i) {
            const uint64_t dai = da + (uint64_t)(i * a16 + kk * 2), dbk = db + (uint64_t)(kk * 2);
            if (i == 1 && kk == 0 && fresh) {   // level 8's first product overwrites
                tc_mma(tmem + (uint32_t)F64_N, dai, dbk, bf16_idesc_mn(F64_M, (F64_SL - 1) * F64_N), 1u);
                tc_mma(tmem + (uint32_t)(8 * F64_N), dai, dbk + (uint64_t)((7 * F64_B_TILE) >> 4), bf16_idesc_mn(F64_M, F64_N), 0u);
            } else {
                tc_mma(tmem + (uint32_t)(i * F64_N), dai, dbk,
                       bf16_idesc_mn(F64_M, (F64_LEV - i < F64_SL ? F64_LEV - i : F64_SL) * F64_N),
                       i == 0 && kk == 0 && fresh ? 0u : 1u);
            }
            if (kk == 1 && i == 3) between();
        }
    }
}

}  // namespace wpccc
