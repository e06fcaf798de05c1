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
// Fixed point: the four differences share the largest one's exponent, its
// leading bit at bit 58, so each carries at least 6 bits more than its own
// double and is cut at 2^-58 of the largest.  Each smoothness indicator is
// normalised on its own (63 bits and an exponent), so that small indicators keep
// their relative precision: a small stencil's weight error only multiplies
// that stencil's equally small candidate.  Weights and their sum are normalised to
// 62 bits, the quotient comes from a reciprocal refined by one third-order
// step.  The total error is below 2^-55 of the largest difference, under the
// rounding of the final addition: against quadruple precision the largest error
// over rough, smooth, jump and flat data is 0.60 of that of the FP64 form it
// replaces, and never larger.
#pragma once
#include <stdint.h>

namespace qlbm {

// Mantissa of a double as a signed fixed-point number, bit 58 the leading bit
// of exponent field E (E >= the value's own field, E >= 1).
__device__ __forceinline__ int64_t i64_fix_(double x, int E)
{
    const uint32_t hi = uint32_t(__double2hiint(x)), lo = uint32_t(__double2loint(x));
    const int e = int((hi >> 20) & 0x7FFu);
    const uint32_t mh = (hi & 0xFFFFFu) | (e ? 0x100000u : 0u);
    const uint64_t m = (((uint64_t(mh) << 32) | lo) << 11) >> min(E - max(e, 1) + 5, 63);
    const int64_t s = int64_t(int32_t(hi) >> 31);
    return (int64_t(m) ^ s) - s;
}

// double(Q) rounded to nearest (ties away), |Q| < 2^62; the conversion instruction
// occupies the FP64 pipe for about 100 cycles per warp, this about 30 issue slots.
__device__ __forceinline__ double i64_to_double_(int64_t Q)
{
    uint64_t q = uint64_t(Q < 0 ? -Q : Q);
    const int sh = min(__clzll(int64_t(q)), 64) - 1;
    q = (q << sh) + 0x200;  // leading bit 62, or 63 after a carry (which the addition below puts in the exponent)
    const uint64_t m = q >> 10;
    const uint32_t hi = uint32_t(m >> 32) + (uint32_t(1084 - sh) << 20);
    return __hiloint2double(Q == 0 ? 0 : int(hi | (uint32_t(Q >> 32) & 0x80000000u)), Q == 0 ? 0 : int(uint32_t(m)));
}

// s^2 + (39/64) d^2 as B 2^-e with B in [2^63, 2^64); zero becomes 2^63 2^-157,
// far below every nonzero one that it is compared with.
__device__ __forceinline__ void i64_indicator_(int64_t s, int64_t d, uint64_t &B, unsigned &e)
{
    uint64_t us = uint64_t(s < 0 ? -s : s), ud = uint64_t(d < 0 ? -d : d);
    const int sh = __clzll(int64_t(us | ud)) - 1;  // |s|, |d| < 2^61
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
    const uint32_t kAbs = 0x7FFFFFFFu;
    int E[N];
    int64_t xa[N], xb[N], xg[N], xc[N];
    uint64_t B[3][N], W[3][N], S[N];
    unsigned e[3][N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const uint32_t m = max(max(uint32_t(__double2hiint(a[k])) & kAbs, uint32_t(__double2hiint(b[k])) & kAbs),
                               max(uint32_t(__double2hiint(g[k])) & kAbs, uint32_t(__double2hiint(c[k])) & kAbs));
        E[k] = max(int(m >> 20), 1);
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
        xa[k] = i64_fix_(a[k], E[k]);
        xb[k] = i64_fix_(b[k], E[k]);
        xg[k] = i64_fix_(g[k], E[k]);
        xc[k] = i64_fix_(c[k], E[k]);
    }
#pragma unroll
    for (int k = 0; k < N; ++k) i64_indicator_(xa[k] + xb[k] + (xb[k] >> 2) + (xb[k] >> 3), xb[k], B[0][k], e[0][k]);
#pragma unroll
    for (int k = 0; k < N; ++k) i64_indicator_(xg[k] - (xb[k] >> 1) - (xb[k] >> 3), xb[k], B[1][k], e[1][k]);
#pragma unroll
    for (int k = 0; k < N; ++k) i64_indicator_(xc[k] - xg[k] - (xg[k] >> 2) - (xg[k] >> 3), xg[k], B[2][k], e[2][k]);
    // products of two indicators, squared, relative to the smallest indicator's
    // exponent: 1 : 6 : 3 are the ideal weights
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const unsigned em = max(max(e[0][k], e[1][k]), e[2][k]);
        const uint64_t M23 = __umul64hi(B[1][k], B[2][k]), M13 = __umul64hi(B[0][k], B[2][k]),
                       M12 = __umul64hi(B[0][k], B[1][k]);
        W[0][k] = __umul64hi(M23, M23) >> min(2u * (em - e[0][k]) + 5u, 63u);
        W[1][k] = 6 * (__umul64hi(M13, M13) >> min(2u * (em - e[1][k]) + 5u, 63u));
        W[2][k] = 3 * (__umul64hi(M12, M12) >> min(2u * (em - e[2][k]) + 5u, 63u));
        S[k] = W[0][k] + W[1][k] + W[2][k];  // in [2^55, 2^62.4)
    }
    int64_t Nm[N], d[N];
    uint64_t x0[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int n = __clz(int(S[k] >> 32)) - 1;
        S[k] <<= n;
        Nm[k] = __mul64hi(int64_t(W[0][k] << n), 2 * xa[k] + 5 * xb[k]) +
                __mul64hi(int64_t(W[1][k] << n), xb[k] + 2 * xg[k]) + __mul64hi(int64_t(W[2][k] << n), 4 * xg[k] - xc[k]);
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
        // Q = 3 (h - f0) 2^(58 - (E - 1023)): one third of the unit, by its exponent
        const int64_t Q = __mul64hi(Nm[k] << 2, X);
        const int unit = E[k] >= 61 ? 0x3FD55555 + ((E[k] - 1081) << 20) : 0;
        h[k] = fma(i64_to_double_(Q), __hiloint2double(E[k] == 0x7FF ? 0x7FF80000 : unit, 0x55555555), f0[k]);
    }
}
__device__ __forceinline__ double weno5_face_i64(double a, double b, double g, double c, double f0)
{
    double h[1];
    weno5_faces_i64<1>({a}, {b}, {g}, {c}, {f0}, h);
    return h[0];
}

}  // namespace qlbm
