// Velocity sets without compiled tiles (any even Q up to kLargeMaxQ; the paper's
// near-ballistic runs use Q = 200), FP64: initial state, densities and output fields
// with the set's tables in device memory.  Their stages are those of
// fdlb_cells.cuh.  Included by the FP64 translation unit only.
#pragma once

#include "qlbm_internal.h"

namespace qlbm {

struct LqTab {
    const double *p, *G, *ca, *cb;
};
__device__ __forceinline__ LqTab lq_tab(const double *tab, int Q)
{
    return LqTab{tab, tab + 3 * Q, tab + 3 * Q + Q * Q, tab + 4 * Q + Q * Q};
}

// Densities of the interior cells for the ball average (balls wider than
// kCellBall): the groups and order of the cell kernel's mass sum.
__global__ void lq_density_kernel(const double2 *__restrict__ psi, int64_t nx, int64_t stride, int Q, int gpairs,
                                  double *__restrict__ n)
{
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= nx) return;
    const int H = Q / 2;
    double acc = 0.0;
    for (int g = 0; g < H; g += gpairs) {
        double part = 0.0;
#pragma unroll 4
        for (int j = g; j < min(H, g + gpairs); ++j)
            part += psi[int64_t(H + j) * stride + kHalo + i].x + psi[int64_t(H - 1 - j) * stride + kHalo + i].x;
        acc += part;
    }
    n[i] = acc;
}

// Discrete equilibrium of given fields at every column (Eq. feq), FP64.
__global__ void lq_init_kernel(const double *__restrict__ rho, const double *__restrict__ u,
                               const double *__restrict__ T, double2 *__restrict__ psi, int64_t nx, int64_t stride,
                               int Q, const double *__restrict__ tab)
{
    const int64_t ncol = nx + 2 * kHalo;
    const int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (c >= ncol) return;
    const LqTab tb = lq_tab(tab, Q);
    const double uu = u[c], TT = T[c], n = rho[c], Tm1 = TT - 1.0;
    for (int k = 0; k < Q; ++k) {
        const double *G = tb.G + int64_t(k) * Q;
        double cm2 = 1.0, cm1 = uu, g = G[0] + G[1] * uu;
        for (int l = 2; l < Q; ++l) {
            const double cl = fma(tb.ca[l] * uu, cm1, tb.cb[l] * Tm1 * cm2);
            g = fma(G[l], cl, g);
            cm2 = cm1;
            cm1 = cl;
        }
        psi[int64_t(k) * stride + c] = make_double2(n * g, 2.0 * TT * n * g);
    }
}

// Output fields and per-block totals, as fdlb_moments_kernel (FP64) with the
// velocity-set size at run time.
__global__ void __launch_bounds__(kMomThreads) lq_fields_kernel(MomentArgs a, int Q, const double *__restrict__ tab)
{
    __shared__ double red[3][kMomThreads];
    const double2 *__restrict__ psi = static_cast<const double2 *>(a.psi);
    const int64_t i = int64_t(blockIdx.x) * kMomThreads + threadIdx.x;
    double M = 0, Pm = 0, E = 0;
    if (i < a.nx) {
        double S0 = 0, S1 = 0, S2 = 0, S3 = 0, R0 = 0, R1 = 0;
        for (int k = 0; k < Q; ++k) {
            const double2 v = psi[int64_t(k) * a.stride + kHalo + i];
            const double p = tab[k];
            S0 += v.x;
            S1 += p * v.x;
            S2 += p * p * v.x;
            S3 += p * p * p * v.x;
            R0 += v.y;
            R1 += p * v.y;
        }
        const double n = S0, u = S1 / n;
        const double c2 = S2 - u * S1;
        const double T = (c2 + R0) / (3.0 * n);
        const double q = 0.5 * (S3 - 3.0 * u * S2 + 2.0 * u * u * S1 + R1 - u * R0);
        const double eta = a.eta0 * n * a.inv_rho_ref;
        const double chi = 0.5 * (2.0 - eta) / ((1.0 - eta) * (1.0 - eta) * (1.0 - eta));
        if (a.rho) a.rho[i] = n;
        if (a.u) a.u[i] = u;
        if (a.T) a.T[i] = T;
        if (a.P) a.P[i] = n * T * (1.0 + 4.0 * eta * chi);
        if (a.q) a.q[i] = q;
        if (a.Pxx) a.Pxx[i] = c2;
        if (!(n > 0.0) || !(T > 0.0) || !isfinite(u) || !isfinite(q)) atomicOr(a.err, 1u);
        M = S0 * a.dx;
        Pm = S1 * a.dx;
        E = 0.5 * (S2 + R0) * a.dx;
    }
    red[0][threadIdx.x] = M;
    red[1][threadIdx.x] = Pm;
    red[2][threadIdx.x] = E;
    __syncthreads();
    for (int h = kMomThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h)
            for (int c = 0; c < 3; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x < 3) a.partial[blockIdx.x * 3 + threadIdx.x] = red[threadIdx.x][0];
}

cudaError_t launch_lq_density(int Q, const void *psi, int64_t nx, int64_t stride, double *n, cudaStream_t s)
{
    lq_density_kernel<<<unsigned((nx + 127) / 128), 128, 0, s>>>(static_cast<const double2 *>(psi), nx, stride, Q,
                                                                 (Q / 2 + kCellWarps - 1) / kCellWarps, n);
    return cudaGetLastError();
}

cudaError_t launch_lq_init(int Q, const double *rho, const double *u, const double *T, void *psi, int64_t nx,
                           int64_t stride, const double *tab, cudaStream_t s)
{
    const int64_t ncol = nx + 2 * kHalo;
    lq_init_kernel<<<unsigned((ncol + 127) / 128), 128, 0, s>>>(rho, u, T, static_cast<double2 *>(psi), nx, stride, Q,
                                                               tab);
    return cudaGetLastError();
}

cudaError_t launch_lq_moments(int Q, const MomentArgs &a, const double *tab, cudaStream_t s)
{
    lq_fields_kernel<<<unsigned(moment_blocks(a.nx)), kMomThreads, 0, s>>>(a, Q, tab);
    return cudaGetLastError();
}

}  // namespace qlbm
