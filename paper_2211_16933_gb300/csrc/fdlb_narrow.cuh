// FP32 stage kernel of small domains: a CTA of 8 warps on 30 cells, the velocity
// pairs dealt to the warps.
//
// The tile kernels (fdlb_kernels.cuh) give each warp its own 31 cells and every
// velocity pair of them, so a domain of 8192 cells is 34 CTAs on 152 SMs and a
// stage is one thread's walk through staging, moments, coefficients and 16 pairs
// (11.6 us).  Here 30 cells share a CTA, the walk is Q / 16 pairs long and 274 CTAs
// cover that domain.  Each warp repeats the cells' collision coefficients and
// Hermite recurrence (about two pairs' worth of instructions), which is what the
// tile kernels win with once the domain fills the GPU.  Measured, us per step (tiles,
// this): Q = 32, 1600 cells 37.0, 13.7; 8192 cells 34.8, 16.5; 16384 cells 36.3, 26.8;
// 24576 cells 36.0, 35.0; 32768 cells 37.1, 44.8.  Q = 8: 1600 cells 14.5, 10.3; 8192
// cells 14.4, 10.8; 32768 cells 16.4, 22.6.  chi_RET-FM averages the
// densities of the staged cells itself from the previous stage's (balls of up to
// kNarrowBall cells), which takes the ball-average launch out of every stage.
// 30 cells and not 31: the same 31 faces, and no warp has more than one strip.
//
// The arithmetic of each cell is that of the tile kernels, in the same order
// (shared functions and sums), and gives the same bits.
#pragma once
#include "fdlb_aux.cuh"
#include "fdlb_kernels.cuh"

namespace qlbm {

constexpr int kNarrowCellsPerCta = 30;

template <int Q, int STAGE, bool RET>
__global__ void __launch_bounds__(kThreads, 2) fdlb_narrow_kernel(NarrowArgs s)
{
    using V = float2;
    using Real = float;
    constexpr TabView TV = tab_view(Q);
    constexpr int H = Q / 2, TILE = kNarrowCellsPerCta, SEG = TILE + 2 * kHalo;
    constexpr int GRP = SumGroup<Real>::pairs, NG = (H + GRP - 1) / GRP;  // moment groups
    constexpr int NP = (H + kWarps - 1) / kWarps;                        // velocity pairs per warp
    static_assert(2 * NG <= kWarps && SEG <= 64, "two warps per moment group");
    __shared__ V s_psi[Q][SEG];
    __shared__ Real s_part[6][NG][SEG];
    __shared__ Real s_n[SEG], s_u[SEG], s_T[SEG], s_q[SEG], s_lnn[SEG], s_lnT[SEG];
    __shared__ Real s_chi[RET ? SEG : 1], s_lnchi[RET ? SEG : 1], s_dn[RET ? H : 1][RET ? 32 : 1];
    __shared__ Real s_bn[RET ? SEG + 2 * kNarrowBall : 1], s_bk[RET ? 2 * kNarrowBall + 1 : 1];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const StageArgs &a = s.a;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t i0 = int64_t(blockIdx.x) * TILE, stride = a.stride;
    const V *__restrict__ in = static_cast<const V *>(a.in);

    // staged cell c (cell i0 - kHalo + c) sits at column i0 + c of its row
    constexpr int LOADS = (Q * SEG + kThreads - 1) / kThreads;
    V ld[LOADS];
#pragma unroll
    for (int k = 0; k < LOADS; ++k) {
        const int e = t + k * kThreads, r = e / SEG;
        if (e < Q * SEG) ld[k] = in[r * stride + i0 + (e - r * SEG)];
    }
    // psi^n of this warp's velocity pairs, used at the very end
    const int st = lane + 3;  // staged cell: lane l computes its right face, lanes 1 .. 30 update it
    const int64_t i = i0 + lane - 1, col = kHalo + i;
    const bool owner = lane >= 1 && lane <= TILE && i < a.nx;
    V bp[NP], bm[NP];
    if (STAGE >= 2) {
        const V *__restrict__ base = static_cast<const V *>(a.base);
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int j = warp + k * kWarps;
            bp[k] = bm[k] = sp2(0.f);
            if (j < H) {
                bp[k] = base[int64_t(H + j) * stride + col];
                bm[k] = base[int64_t(H - 1 - j) * stride + col];
            }
        }
    }
    if (RET && t >= kThreads - 64) {
        // nbar as fdlb_fm_kernel forms it, then Eq. (chi_ret), by two warps while the loads above are in
        // flight.  The ball's weights (one FP64 conversion each) and densities go through shared memory: with
        // each thread fetching and converting all of its own, balls of 8 and 16 cells were slower than on
        // tiles with the average as a launch of its own (us per step; tiles, each its own, this: Q = 8, 16384 cells, 16 cells:
        // 24.6, 52.7, 23.5; Q = 20, 5000 cells, 8 cells: 34.8, 30.8, 18.5).  A ball within its cell has one
        // weight and needs no trip through shared memory (balls of one cell are faster with it).
        const int c = t - (kThreads - 64), W = s.f.W;
        const Real *n = static_cast<const Real *>(s.f.n);
        Real nbar = 0.f;
        if (W == 0) {
            if (c < SEG) nbar = fma_(Real(s.f.K[0]), fm_density<Real>(s.f, n, i0 - kHalo + c), nbar);
        } else {
            const double weight = s.f.K[min(c, 2 * W)];  // in flight beside the densities
            for (int e = c; e < SEG + 2 * W; e += 64) s_bn[e] = fm_density<Real>(s.f, n, i0 - kHalo - W + e);
            if (c <= 2 * W) s_bk[c] = Real(weight);
            asm volatile("bar.sync 1, 64;" ::: "memory");
            if (c < SEG)
#pragma unroll 4
                for (int d = 0; d <= 2 * W; ++d) nbar = fma_(s_bk[d], s_bn[c + d], nbar);
        }
        if (c < SEG) {
            const Real chi = chi_of_nbar_(a, nbar);
            s_chi[c] = chi;
            s_lnchi[c] = log_(chi);
        }
    }
#pragma unroll
    for (int k = 0; k < LOADS; ++k) {
        const int e = t + k * kThreads, r = e / SEG;
        if (e < Q * SEG) s_psi[r][e - r * SEG] = ld[k];
    }
    __syncthreads();

    // moments: group g of 8 velocity pairs by warps 2 g (cells 0 .. 31) and 2 g + 1
    const bool ff = !QL_F32_SUMS_FP64 && !a.sums64;
    {
        const int g = warp >> 1, c = (warp & 1) * 32 + lane;
        if (g < NG && c < SEG) {
            GroupSums<Real> gs;
#pragma unroll
            for (int k = 0; k < GRP; ++k) {
                const int j = g * GRP + k;
                if (j < H)
                    gs.add(QL_TAB[TV.p + H + j], QL_TAB[TV.p2 + H + j], QL_TAB[TV.p3 + H + j], s_psi[H + j][c],
                           s_psi[H - 1 - j][c]);
            }
            s_part[0][g][c] = gs.s01.x;
            s_part[1][g][c] = gs.s01.y;
            s_part[2][g][c] = gs.s11.x;
            s_part[3][g][c] = gs.s11.y;
            s_part[4][g][c] = gs.s2;
            s_part[5][g][c] = gs.s3;
        }
    }
    __syncthreads();
    if (t < SEG) {
        MomentSums<Real> ms;
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            GroupSums<Real> gs;
            gs.s01 = mk2(s_part[0][g][t], s_part[1][g][t]);
            gs.s11 = mk2(s_part[2][g][t], s_part[3][g][t]);
            gs.s2 = s_part[4][g][t];
            gs.s3 = s_part[5][g][t];
            ms.add(gs, ff);
        }
        Real n, u, T, q;
        ms.finish(ff, n, u, T, q);
        const int64_t ci = i0 - kHalo + t;
        if (ci >= 0 && ci < a.nx && nonphysical_(n, u, T, q)) atomicOr(a.err, 1u);
        s_n[t] = n;
        s_u[t] = u;
        s_T[t] = T;
        s_q[t] = q;
        s_lnn[t] = log_(n);
        s_lnT[t] = log_(T);
    }
    __syncthreads();

    if (warp < H) {
        const Real inv_dx = Real(a.inv_dx), u = s_u[st], T = s_T[st];
        const CellCoefs<Real> cc = cell_coefs_<Real, RET>(
            a, STAGE, s_n[st], u, T, s_q[st], cd6_(s_lnn, st) * inv_dx, cd6_(s_u, st) * inv_dx, cd6_(s_lnT, st) * inv_dx,
            RET ? s_chi[RET ? st : 0] : 0.f, RET ? cd6_(s_lnchi, RET ? st : 3) * inv_dx : 0.f);
        const V D0 = cc.D0, D1 = cc.D1, D2 = cc.D2, D3 = cc.D3, kpsi = sp2(cc.kpsi);
        // Hermite coefficients d_l = l! c_l, as in the tile kernels
        V ch[H];
        Real cm2 = 1.f, cm1 = u;
        ch[0] = mk2(cm2, cm1);
        const Real Tm1 = T - 1.f;
#pragma unroll
        for (int m = 1; m < H; ++m) {
            const Real ce = fma_(u, cm1, (QL_TAB[TV.cb + 2 * m] * Tm1) * cm2);
            const Real co = fma_(u, ce, (QL_TAB[TV.cb + 2 * m + 1] * Tm1) * cm1);
            ch[m] = mk2(ce, co);
            cm2 = ce;
            cm1 = co;
        }
        const Real adv = advection_<Real>(a, STAGE);
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int j = warp + k * kWarps;
            if (j >= H) break;
            const V *rp = s_psi[H + j], *rm = s_psi[H - 1 - j];
            const V fp0 = rp[st], fm0 = rm[st];
            const V hp = weno5_face2<Real>(rp[st - 2], rp[st - 1], fp0, rp[st + 1], rp[st + 2]);
            const V hm = weno5_face2<Real>(rm[st + 3], rm[st + 2], rm[st + 1], fm0, rm[st - 1]);
            const V hpl = mk2(__shfl_up_sync(0xffffffffu, hp.x, 1), __shfl_up_sync(0xffffffffu, hp.y, 1));
            const V hml = mk2(__shfl_up_sync(0xffffffffu, hm.x, 1), __shfl_up_sync(0xffffffffu, hm.y, 1));
            V eo = sp2(0.f);
            const V *Gj = reinterpret_cast<const V *>(&QL_TAB[TV.G + (H + j) * Q]);
#pragma unroll
            for (int m = 0; m < H; ++m) eo = fma2(Gj[m], ch[m], eo);
            const Real gpv = eo.x + eo.y, gmv = eo.x - eo.y, p = QL_TAB[TV.p + H + j];
            const V padv = sp2(p * adv), p2 = sp2(QL_TAB[TV.p2 + H + j]);
            const V E = fma2(D2, p2, D0);
            const V O = mul2(fma2(D3, p2, D1), sp2(p));
            const V Pp = add2(E, O), Pm = sub2(E, O);
            V op = fma2(padv, sub2(hpl, hp), fma2(fp0, kpsi, mul2(sp2(gpv), Pp)));
            V om = fma2(padv, sub2(hm, hml), fma2(fm0, kpsi, mul2(sp2(gmv), Pm)));
            if (STAGE >= 2) {
                const V c = sp2(1.f - rk_weight_<Real>(STAGE));
                op = fma2(c, bp[k], op);
                om = fma2(c, bm[k], om);
            }
            if (owner) {
                V *qp = static_cast<V *>(a.out) + int64_t(H + j) * stride + col;
                V *qm = static_cast<V *>(a.out) + int64_t(H - 1 - j) * stride + col;
                *qp = op;
                *qm = om;
                if (STAGE != 0 && a.periodic) {  // periodic images in the ghost columns
                    if (i < kHalo) {
                        qp[a.nx] = op;
                        qm[a.nx] = om;
                    }
                    if (i >= a.nx - kHalo) {
                        qp[-a.nx] = op;
                        qm[-a.nx] = om;
                    }
                }
            }
            if (RET && STAGE != 0) s_dn[RET ? j : 0][RET ? lane : 0] = op.x + om.x;
        }
    }
    if (RET && STAGE != 0) {
        // density of the output, summed over the pairs in the tile kernels' order
        __syncthreads();
        if (warp == 0 && owner) {
            Real acc = 0.f;
#pragma unroll
            for (int j = 0; j < H; ++j) acc += s_dn[RET ? j : 0][RET ? lane : 0];
            static_cast<Real *>(a.nout)[i] = acc;
        }
    }
}

template <int Q, bool RET>
static cudaError_t narrow_q(int stage, const NarrowArgs &s, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned((s.a.nx + kNarrowCellsPerCta - 1) / kNarrowCellsPerCta));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    // programmatic stream serialisation, as for the tile kernels
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    switch (stage) {
    case 0: return cudaLaunchKernelEx(&cfg, fdlb_narrow_kernel<Q, 0, RET>, s);
    case 1: return cudaLaunchKernelEx(&cfg, fdlb_narrow_kernel<Q, 1, RET>, s);
    case 2: return cudaLaunchKernelEx(&cfg, fdlb_narrow_kernel<Q, 2, RET>, s);
    case 3: return cudaLaunchKernelEx(&cfg, fdlb_narrow_kernel<Q, 3, RET>, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_narrow_f32(int Q, int stage, const NarrowArgs &s, bool ret, cudaStream_t st)
{
    if (ret && (!s.f.n || s.f.W > kNarrowBall || (stage != 0 && !s.a.nout))) return cudaErrorInvalidValue;
    switch (Q) {
    case 8: return ret ? narrow_q<8, true>(stage, s, st) : narrow_q<8, false>(stage, s, st);
    case 16: return ret ? narrow_q<16, true>(stage, s, st) : narrow_q<16, false>(stage, s, st);
    case 20: return ret ? narrow_q<20, true>(stage, s, st) : narrow_q<20, false>(stage, s, st);
    case 24: return ret ? narrow_q<24, true>(stage, s, st) : narrow_q<24, false>(stage, s, st);
    case 32: return ret ? narrow_q<32, true>(stage, s, st) : narrow_q<32, false>(stage, s, st);
    case 40: return ret ? narrow_q<40, true>(stage, s, st) : narrow_q<40, false>(stage, s, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace qlbm
