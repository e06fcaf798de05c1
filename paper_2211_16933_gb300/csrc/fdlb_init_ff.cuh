// FP32 state of the discrete equilibrium of given fields: fdlb_init_kernel's sums
// in double-FP32 (about 48 bits), rounded once to FP32.
//
// fdlb_init_kernel<float> was bound by the FP64 pipe (about 64 cycles per warp
// instruction and sub-partition): 518 FP64 instructions per cell at Q = 24, 922 us for 10^6
// cells where the 0.2 GB written take 29 (a ql_load_fields call with three steps after it: 2466
// us, now 1707).  Here a term of the sums is 12 packed FP32
// instructions for an even and an odd coefficient together: the exact product's two halves,
// the error-free sum, and the low parts in a second accumulator (compensated dot
// product, T. Ogita, S. M. Rump, S. Oishi, SIAM J. Sci. Comput. 26, 2005).  Fields outside
// the range in which its intermediate values stay far from FP32's limits (|u|, |T - 1|
// < 8, n and T neither tiny nor huge) take the FP64 sums.  So do velocity pairs with a g below 2^-12 of
// the sum of its terms' magnitudes (fast velocities of states far from u = 0, T = 1), where about 48 bits
// are too few: against quadruple precision the largest error there was 2 to 10^3 times that of the
// FP64 sums, and above the line it is 0.5001 FP32 units in the last place, as theirs (0.5000; 240000 random
// states, all velocity sets).  None are below it for |u| < 0.1 and |T - 1| < 0.05; at Q = 32, |u| < 0.4 and |T - 1|
// < 0.2 6 % are, u = 1.0 to 1.4 and T = 0.4 to 0.6 47 %.
#pragma once
#include "fdlb_aux.cuh"

namespace qlbm {

// Per velocity set: rows of (Gh[2m], Gh[2m+1], -Gl[2m], -Gl[2m+1]) for the velocities p > 0,
// then (ca, cb) as (h, l, h, l) per coefficient.
QL_HD constexpr int ff_tab_size(int Q) { return Q / 2 * (Q / 2) + Q; }
QL_HD constexpr int ff_tab_offset(int Q)
{
    // tables of the sizes in kQList, in ascending order
    return (Q > 8 ? ff_tab_size(8) : 0) + (Q > 16 ? ff_tab_size(16) : 0) + (Q > 20 ? ff_tab_size(20) : 0) +
           (Q > 24 ? ff_tab_size(24) : 0) + (Q > 32 ? ff_tab_size(32) : 0) + (Q > 40 ? ff_tab_size(40) : 0);
}
constexpr int kFfTabTotal = ff_tab_offset(1 << 30);
static __constant__ float4 QL_FFTAB[kFfTabTotal];

static cudaError_t upload_ff_table(const double *all)
{
    static float4 host[kFfTabTotal];
    auto low = [](double v) { return float(v - double(float(v))); };
    for (int k = 0; k < kNumQ; ++k) {
        const int Q = kQList[k], H = Q / 2;
        const TabView tv = tab_view(Q);
        float4 *T = host + ff_tab_offset(Q);
        for (int j = 0; j < H; ++j)
            for (int m = 0; m < H; ++m) {
                const double *G = all + tv.G + (H + j) * Q + 2 * m;
                T[j * H + m] = make_float4(float(G[0]), float(G[1]), -low(G[0]), -low(G[1]));
            }
        for (int l = 0; l < Q; ++l) {
            const double a = l >= 2 ? all[tv.ca + l] : 0.0, b = l >= 2 ? all[tv.cb + l] : 0.0;
            T[H * H + l] = make_float4(float(a), low(a), float(b), low(b));
        }
    }
    return cudaMemcpyToSymbol(QL_FFTAB, host, sizeof(host));
}

// Exponent of |x| (1024 for infinities and NaN).
__device__ __forceinline__ int exponent_(double x) { return ((__double2hiint(x) >> 20) & 0x7FF) - 1023; }
// x as double-FP32 to 2^-48 of |x|, by integer operations, for exponents of -90 to 60; smaller values
// give zero.
__device__ __forceinline__ FF ff_split(double x)
{
    const int hi = __double2hiint(x), lo = __double2loint(x), e = exponent_(x);
    if (e < -90) return {0.f, 0.f};
    const unsigned top = unsigned((hi & 0xFFFFF) | 0x100000) << 3 | unsigned(lo) >> 29;
    const float s = __int_as_float(((e - 23 + 127) << 23) | (hi & 0x80000000));
    return fast_two_sum(float(top) * s, float(unsigned(lo) & 0x1FFFFFFFu) * (s * 0x1p-29f));
}

// FP64 sums of the velocity pairs whose bit in `pairs` is set, as init_column (threads that skipped
// different pairs went through the loop one after the other: 10.1 ms for 10^6 cells at Q = 40, u = 1.0 to
// 1.4 and T = 0.4 to 0.6, 1.9 so, all in FP64 2.2).
template <int Q>
__device__ __noinline__ void init_pairs_f64(double uu, double TT, double n, float2 *__restrict__ psi, int64_t stride,
                                            const double *__restrict__ tab, unsigned pairs)
{
    init_column<float, Q>(uu, TT, n, psi, stride, tab, __reduce_or_sync(__activemask(), pairs), pairs);
}

// One thread per column, as fdlb_init_kernel.
template <int Q>
__global__ void __launch_bounds__(256) fdlb_init_ff_kernel(const double *__restrict__ rho,
                                                           const double *__restrict__ u, const double *__restrict__ T,
                                                           float2 *__restrict__ psi, int64_t nx, int64_t stride,
                                                           const double *__restrict__ tab)
{
    constexpr int H = Q / 2, OFF = ff_tab_offset(Q);
    const int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;  // column, cell c - kHalo
    if (c >= nx + 2 * kHalo) return;
    const double uu = u[c], TT = T[c], n = rho[c], Tm = TT - 1.0;
    const int en = exponent_(n), et = exponent_(TT);
    if (!(exponent_(uu) < 3 && exponent_(Tm) < 3 && en >= -60 && en < 60 && et >= -60 && et < 60)) {
        init_pairs_f64<Q>(uu, TT, n, psi + c, stride, tab, ~0u);
        return;
    }
    const FF fu = ff_split(uu), ft = ff_split(Tm), fn = ff_split(n);
    FF t2 = ff_split(TT);
    t2 = {t2.h + t2.h, t2.l + t2.l};
    float2 ch[H], cl[H];  // coefficients (2m, 2m + 1), high and low parts
    {
        FF m2 = {1.f, 0.f}, m1 = fu;
        ch[0] = mk2(m2.h, m1.h);
        cl[0] = mk2(m2.l, m1.l);
#pragma unroll
        for (int m = 1; m < H; ++m) {
            const float4 A = QL_FFTAB[OFF + H * H + 2 * m], B = QL_FFTAB[OFF + H * H + 2 * m + 1];
            const FF ce = ff_add(ff_mul(ff_mul({A.x, A.y}, fu), m1), ff_mul(ff_mul({A.z, A.w}, ft), m2));
            const FF co = ff_add(ff_mul(ff_mul({B.x, B.y}, fu), ce), ff_mul(ff_mul({B.z, B.w}, ft), m1));
            ch[m] = mk2(ce.h, co.h);
            cl[m] = mk2(ce.l, co.l);
            m2 = ce;
            m1 = co;
        }
    }
    unsigned steep = 0;  // pairs left to the FP64 sums
#pragma unroll 1
    for (int j = 0; j < H; ++j) {
        float2 s = sp2(0.f), r = sp2(0.f);  // the even and the odd sum: rounded, and what it lacks
        float size = 0.f;                   // sum of the magnitudes
#pragma unroll
        for (int m = 0; m < H; ++m) {
            const float4 g = QL_FFTAB[OFF + j * H + m];
            const float2 gh = mk2(g.x, g.y), ngh = mk2(-g.x, -g.y), ngl = mk2(g.z, g.w);
            const float2 p = mul2(gh, ch[m]);
            size += fabsf(p.x) + fabsf(p.y);
            const float2 lack = fma2(ngl, ch[m], fma2(ngh, cl[m], fma2(ngh, ch[m], p)));  // p - (exact term)
            const float2 w = add2(s, p), b = sub2(w, s);
            r = add2(r, sub2(add2(sub2(s, sub2(w, b)), sub2(p, b)), lack));
            s = w;
        }
        const FF e = two_sum(s.x, r.x), o = two_sum(s.y, r.y);
        const FF sp = ff_add(e, o), sm = ff_add(e, ff_neg(o));
        if (!(fminf(fabsf(sp.h), fabsf(sm.h)) >= 0x1p-12f * size)) steep |= 1u << j;
        const FF gp = ff_mul(fn, sp), gm = ff_mul(fn, sm);
        psi[int64_t(H + j) * stride + c] = mk2(gp.h, ff_mul(t2, gp).h);
        psi[int64_t(H - 1 - j) * stride + c] = mk2(gm.h, ff_mul(t2, gm).h);
    }
    if (steep) init_pairs_f64<Q>(uu, TT, n, psi + c, stride, tab, steep);
}

}  // namespace qlbm
