// WENO-5 face values of double data in 64-bit integer arithmetic.
//
// GB300 issues one FP64 warp instruction per SM sub-partition every 64 to 76
// cycles (measured with 1 and 2 warps each), and a 64 x 64 -> high 64 bit
// product takes about 20.  The nonlinear weights of one face value cost 46
// FP64 instructions (about 3500 cycles), and FP64 arithmetic bounded every
// FP64 kernel of this library (FP64 pipe 86 % busy).  So the five values'
// differences are formed in FP64 (4 instructions), the weights and the
// weighted sum in integers beside the FP64 pipe, and the result is added to f0
// by one fused multiply-add.
//
// Fixed point: the two differences of each stencil share the larger one's exponent, its
// leading bit at bit 59, so each carries at least 7 bits more than its own
// double and is cut at 2^-59 of the stencil's larger one.  Each smoothness indicator is
// normalised on its own (63 bits and an exponent).  The weighted sum is formed in the unit of its
// largest term: a stencil's differences may be 2^k times the smoothest one's, its weight is then about
// 2^-4k of it, so that it stays within a few bits of the smoothest one's unit.  The error is about 2^-54 of the
// differences of the stencils that carry the weight, whatever the other differences are: values far
// smaller than a jump beside them (populations of fast velocities at an unresolved jump) keep their relative
// precision and their sign.  (One exponent for all four differences, the former form, made +-5e-18 of a tail of
// 1e-25 beside a value of 1.)  Weights and their sum are normalised to 62 bits, the
// quotient comes from a reciprocal refined by one third-order step.
// Against quadruple precision, largest and mean error over max(|f0|, |h|) in units of 1e-16, FP64 product form -> this
// (4e6 faces each, the largest difference between a half and twice f0): random data 4.95, 0.402 -> 1.69, 0.370;
// Gaussian profiles 2.29, 0.407 -> 1.65, 0.370; a jump between nearly flat sides 1.42, 0.398 -> 1.18, 0.398; values
// falling by e^5 per cell 3.49, 0.678 -> 1.64, 0.404, rising by e^12 2.68, 0.527 -> 1.82, 0.494; a tail of 1e-25
// beside 1 1.24, 0.461 -> 1.27, 0.460; exponents uniform in e^+-8 4970, 1.03 -> 3310, 0.778.  The exponents per stencil
// cost the tile kernels 3 % (262144 cells, Q = 32: 2944 -> 3038 us per step) and the small-domain kernels nothing, the unit's
// normal range 0.8 % (3036 -> 3060).
#pragma once
#include <stdint.h>

namespace qlbm {

// Exponent field of a double (0 for zero and subnormal numbers).
__device__ __forceinline__ int exp_field_(double x) { return int((uint32_t(__double2hiint(x)) >> 20) & 0x7FFu); }

// Signed mantissa of a double of exponent field e, leading bit 62 (subnormal numbers: that of field 1).
__device__ __forceinline__ int64_t i64_mantissa_(double x, int e)
{
    const uint32_t hi = uint32_t(__double2hiint(x)), lo = uint32_t(__double2loint(x));
    const uint32_t mh = (hi & 0xFFFFFu) | (e ? 0x100000u : 0u);
    const int64_t m = int64_t(((uint64_t(mh) << 32) | lo) << 10), s = int64_t(int32_t(hi) >> 31);
    return (m ^ s) - s;
}
// The same as fixed point, bit 59 the leading bit of exponent field E >= e, E >= 1.
__device__ __forceinline__ int64_t i64_fix_(int64_t m, int e, int E) { return m >> min(E - max(e, 1) + 3, 63); }

// Q 2^-low rounded to nearest (ties away), |Q| < 2^62, 0 <= low < 900; the conversion instruction
// occupies the FP64 pipe for about 100 cycles per warp, this about 30 issue slots.
__device__ __forceinline__ double i64_to_double_(int64_t Q, int low)
{
    uint64_t q = uint64_t(Q < 0 ? -Q : Q);
    const int sh = min(__clzll(int64_t(q)), 64) - 1;
    q = (q << sh) + 0x200;  // leading bit 62, or 63 after a carry (which the addition below puts in the exponent)
    const uint64_t m = q >> 10;
    const uint32_t hi = uint32_t(m >> 32) + (uint32_t(1084 - sh - low) << 20);
    return __hiloint2double(Q == 0 ? 0 : int(hi | (uint32_t(Q >> 32) & 0x80000000u)), Q == 0 ? 0 : int(uint32_t(m)));
}

// s^2 + (39/64) d^2 as B 2^-e with B in [2^63, 2^64); zero becomes 2^63 2^-157,
// far below every nonzero one that it is compared with.
__device__ __forceinline__ void i64_indicator_(int64_t s, int64_t d, uint64_t &B, unsigned &e)
{
    uint64_t us = uint64_t(s < 0 ? -s : s), ud = uint64_t(d < 0 ? -d : d);
    const int sh = __clzll(int64_t(us | ud)) - 1;  // |s|, |d| < 2^62
    us <<= sh;
    ud <<= sh;
    const uint64_t b = __umul64hi(us, us) + __umul64hi(ud, (ud >> 1) + (ud >> 3) - (ud >> 6));
    const int k = min(__clz(int(b >> 32)), 31);  // b >= 2^59 unless both are zero
    B = (b << k) | 0x8000000000000000ull;
    e = unsigned(2 * sh + k);
}

// N face values h[e] = f0 + (sum_q w_q (F^q - f0)) / sum_q w_q of App. A.2 from the
// differences a = f_{i-2} - f_{i-1}, b = f_i - f_{i-1}, g = f_{i+1} - f_i and
// c = f_{i+2} - f_{i+1}, with w_q = delta_q prod_{r != q} beta_r^2 (rows of
// Table weno_x with zero indicators included: weights of zero indicators
// outweigh the others, equal zero indicators share as delta_q).  The
// indicators, up to a common factor, are sums of two squares:
//   (a + 11/8 b)^2 + 39/64 b^2,  (g - 5/8 b)^2 + 39/64 b^2,  (c - 11/8 g)^2 + 39/64 g^2,
// and 6 (F^q - f0) = 2a + 5b, b + 2g, 4g - c.  A non-finite difference gives NaN.
// One face value is a chain of about 600 instructions with little of it independent;
// the N are written side by side, step by step, so that a lone warp has N
// chains in flight (N = 2 in the small-domain kernels, 7 - 10 % of a step; the tile
// kernels, with three warps to an issue slot, run 5 % slower so and take N = 1).
template <int N>
__device__ __forceinline__ void weno5_faces_i64(const double (&a)[N], const double (&b)[N], const double (&g)[N],
                                                const double (&c)[N], const double (&f0)[N], double (&h)[N])
{
    int E[3][N];         // exponent of each stencil
    int64_t x[3][2][N];  // its two differences
    uint64_t B[3][N], W[3][N], S[N];
    unsigned e[3][N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int ea = exp_field_(a[k]), eb = exp_field_(b[k]), eg = exp_field_(g[k]), ec = exp_field_(c[k]);
        E[0][k] = max(max(ea, eb), 1);
        E[1][k] = max(max(eb, eg), 1);
        E[2][k] = max(max(eg, ec), 1);
        const int64_t ma = i64_mantissa_(a[k], ea), mb = i64_mantissa_(b[k], eb), mg = i64_mantissa_(g[k], eg),
                      mc = i64_mantissa_(c[k], ec);
        x[0][0][k] = i64_fix_(ma, ea, E[0][k]);
        x[0][1][k] = i64_fix_(mb, eb, E[0][k]);
        x[1][0][k] = i64_fix_(mb, eb, E[1][k]);
        x[1][1][k] = i64_fix_(mg, eg, E[1][k]);
        x[2][0][k] = i64_fix_(mg, eg, E[2][k]);
        x[2][1][k] = i64_fix_(mc, ec, E[2][k]);
    }
#pragma unroll
    for (int k = 0; k < N; ++k)
        i64_indicator_(x[0][0][k] + x[0][1][k] + (x[0][1][k] >> 2) + (x[0][1][k] >> 3), x[0][1][k], B[0][k], e[0][k]);
#pragma unroll
    for (int k = 0; k < N; ++k)
        i64_indicator_(x[1][1][k] - (x[1][0][k] >> 1) - (x[1][0][k] >> 3), x[1][0][k], B[1][k], e[1][k]);
#pragma unroll
    for (int k = 0; k < N; ++k)
        i64_indicator_(x[2][1][k] - x[2][0][k] - (x[2][0][k] >> 2) - (x[2][0][k] >> 3), x[2][0][k], B[2][k], e[2][k]);
    // products of two indicators, squared, times the ideal weights 1 : 6 : 3; the weight of stencil q is
    // W[q] 2^(h[q] - s[q]) up to a common factor, h = 2 e - 4 E and s = 5, 2, 3, its differences have exponent E
    int T[N], n[N];
    int64_t Nm[N], d[N];
    uint64_t x0[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const uint64_t M23 = __umul64hi(B[1][k], B[2][k]), M13 = __umul64hi(B[0][k], B[2][k]),
                       M12 = __umul64hi(B[0][k], B[1][k]);
        W[0][k] = __umul64hi(M23, M23);
        W[1][k] = 3 * (__umul64hi(M13, M13) >> 2);
        W[2][k] = 3 * (__umul64hi(M12, M12) >> 2);
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int h0 = 2 * int(e[0][k]) - 4 * E[0][k], h1 = 2 * int(e[1][k]) - 4 * E[1][k], h2 = 2 * int(e[2][k]) - 4 * E[2][k];
        const int hm = max(max(h0, h1), h2);
        // the weights' sum relative to the smallest indicator's exponent, in [2^55, 2^62.4)
        S[k] = (W[0][k] >> min(hm - h0 + 5, 63)) + (W[1][k] >> min(hm - h1 + 2, 63)) + (W[2][k] >> min(hm - h2 + 3, 63));
        // 6 times the weighted sum of the candidates times 2^-T: the largest term's weight shifted by 2 (three terms
        // below 2^60.8)
        const int g0 = h0 + E[0][k] - 5, g1 = h1 + E[1][k] - 2, g2 = h2 + E[2][k] - 3;
        const int gm = max(max(g0, g1), g2) + 2;
        T[k] = gm - hm;
        Nm[k] = __mul64hi(int64_t(W[0][k] >> min(gm - g0, 63)), 2 * x[0][0][k] + 5 * x[0][1][k]) +
                __mul64hi(int64_t(W[1][k] >> min(gm - g1, 63)), x[1][0][k] + 2 * x[1][1][k]) +
                __mul64hi(int64_t(W[2][k] >> min(gm - g2, 63)), 4 * x[2][0][k] - x[2][1][k]);
        n[k] = __clz(int(S[k] >> 32)) - 1;
        S[k] <<= n[k];
    }
    // X = 2^125 / S: x0 from the FP32 reciprocal (relative error about 2^-22),
    // then x0 (1 + d + d^2) with d = 1 - S x0 (Householder's third-order step)
#pragma unroll
    for (int k = 0; k < N; ++k) {
        float rf;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(float(uint32_t(S[k] >> 32))));
        // S = 2^62 (one weight, of indicators that are powers of two, outweighs the others) has X =
        // 2^63, which as a signed number turns the correction round: x0 stays below it, and so does X
        x0[k] = uint64_t(min(uint32_t(rf * 2305843009213693952.0f), 0x7FFFFFFFu)) << 32;
        d[k] = int64_t(0x2000000000000000ull - __umul64hi(S[k], x0[k]));
        const int32_t dd = int32_t(d[k] >> 10);
        d[k] += (int64_t(dd) * dd) >> 41;
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int64_t X = int64_t(x0[k] + uint64_t(__mul64hi(d[k] << 20, int64_t(x0[k] >> 1)) >> 16));
        // Q = 6 (h - f0) 2^(1079 - T - n): a sixth of the unit, by its exponent, which is kept in the normal
        // range (T + n is -2 at the least; below 60 only where differences are below 2^-962, or zero)
        const int64_t Q = __mul64hi(Nm[k], X);
        const int m = T[k] + n[k], low = max(60 - m, 0), unit = 0x3FD55555 + ((m + low - 1080) << 20);
        const bool nan = max(max(E[0][k], E[1][k]), E[2][k]) == 0x7FF;
        h[k] = fma(i64_to_double_(Q, low), __hiloint2double(nan ? 0x7FF80000 : unit, 0x55555555), f0[k]);
    }
}
__device__ __forceinline__ double weno5_face_i64(double a, double b, double g, double c, double f0)
{
    double h[1];
    weno5_faces_i64<1>({a}, {b}, {g}, {c}, {f0}, h);
    return h[0];
}

}  // namespace qlbm
