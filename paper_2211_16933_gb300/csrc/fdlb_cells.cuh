// FP64 stage kernels of small domains and of velocity sets without compiled
// tiles: one Runge-Kutta stage as two launches with the per-cell quantities in
// global memory (L2) between them:
//   fdlb_cell_kernel  moments, gradients, collision coefficients and Hermite
//                     coefficients of every cell;
//   fdlb_pair_kernel  one warp per (31 cells, velocity pair): WENO-5 faces,
//                     equilibrium, targets and the update.
// Included by fdlb_f64.cu after the tile kernels.
//
// Why two launches: on a domain of few tiles the tile kernels (fdlb_kernels.cuh)
// keep a handful of SMs busy, each thread walking through the moments, the
// collision coefficients, the Hermite recurrence and all velocity pairs of its
// cell in turn; splitting the pairs over CTAs repeats the per-cell part in each. Here
// both parts are spread: the per-cell part over 8 warps for 26 cells (groups of
// velocity pairs, then the logarithms, the coefficients and the recurrence side
// by side), the rest over (cells / 31) x (Q / 2) warps.  What bounds them is the
// latency of one warp's chain: an FP64 instruction takes 64 cycles of its SM
// sub-partition whatever else runs there.  Measured against the tile kernels with
// the same arithmetic (us per step): 1024 cells, Q = 32: 63 against 113; 4096: 90
// against 162; 65536: 753 against 966; 640 cells, Q = 20, chi_RET-FM: 61 against
// 106; 131072 cells: equal, and the tiles ahead from there on (2.13 against 2.40 ms
// at 262144 cells, Q = 24).  FP32 stages are short enough for the second launch to
// cost more than it gives (Q = 8, 1600 cells: 22.7 against 14.4), so FP32 has no
// such form.  The paper's Q = 200 tube of 160 cells, per stage: 290 us with its
// former kernels (one thread per column for the moments, one recurrence of Q
// steps per velocity), 61 us so.
//
// The arithmetic of each quantity is that of the tile kernels, in the same
// order (shared functions), so tiled velocity sets give the same bits on either path.
#pragma once
#include "fdlb_kernels.cuh"

namespace qlbm {

constexpr int kCellWarps = 8;   // warps of fdlb_cell_kernel; also its most groups of velocity pairs
constexpr int kPairWarps = 4;   // velocity pairs per block of fdlb_pair_kernel
constexpr int kPairCells = 31;  // cells per warp; lane 0 computes the left face

// Velocity-set tables: the kernels' constant bank (tiled sets), or device memory
// laid out as tab_view with offset 0 (other sets: FP64, normalised coefficients).
template <bool LQ>
struct SetTables {
    const double *lq;
    TabView tv;
    __device__ __forceinline__ SetTables(const CellArgs &s)
        : lq(LQ ? s.tab : nullptr), tv(LQ ? tab_view0(s.Q) : tab_view(s.Q))
    {
    }
    __device__ __forceinline__ double at(int e) const { return LQ ? lq[e] : QL_TAB[e]; }
    __device__ __forceinline__ double2 pair(int e) const
    {
        return LQ ? *reinterpret_cast<const double2 *>(lq + e) : *reinterpret_cast<const double2 *>(&QL_TAB[e]);
    }
};

// Cell whose column holds the state of cell i: its periodic image, or the cell
// itself with the outermost ghost columns repeated beyond them.
__device__ __forceinline__ int64_t source_cell_(int64_t i, int64_t nx, bool periodic)
{
    if (i >= 0 && i < nx) return i;
    if (periodic) return ((i % nx) + nx) % nx;
    return i < -kHalo ? -kHalo : (i > nx + kHalo - 1 ? nx + kHalo - 1 : i);
}

// Block b computes cells b ncell .. with one cell per lane and `halo` cells more
// on each side (3 for the gradients; with chi_RET-FM and a ball of W <=
// kCellBall cells W more, whose densities it averages itself; wider balls read
// nbar from a.nbar).
template <bool RET, bool LQ>
__global__ void __launch_bounds__(32 * kCellWarps) fdlb_cell_kernel(CellArgs s)
{
    using V = double2;
    __shared__ double s_part[6][kCellWarps][32];
    __shared__ double s_sum[7][32];
    constexpr int kChunk = 16;
    __shared__ double s_fac[LQ ? 2 : 1][2][kChunk][32];
    __shared__ double s_n[32], s_u[32], s_T[32], s_q[32], s_lnn[32], s_lnT[32], s_chi[32], s_lnchi[32];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const StageArgs &a = s.a;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, H = s.Q / 2;
    const SetTables<LQ> tab(s);
    const TabView tv = tab.tv;
    const bool inball = RET && s.W <= kCellBall;
    const int halo = 3 + (inball ? s.W : 0), ncell = 32 - 2 * halo;
    const int64_t i = s.i0 + int64_t(blockIdx.x) * ncell - halo + lane;
    const bool own = lane >= halo && lane < 32 - halo && i < s.i1;

    // groups of `gpairs` velocity pairs, one warp each (at most kCellWarps groups)
    if (warp * s.gpairs < H) {
        const V *__restrict__ psi = static_cast<const V *>(a.in) + kHalo + source_cell_(i, a.nx, a.periodic != 0);
        const int j1 = min(H, (warp + 1) * s.gpairs);
        GroupSums<double> g;
#pragma unroll 4
        for (int j = warp * s.gpairs; j < j1; ++j)
            g.add(tab.at(tv.p + H + j), tab.at(tv.p2 + H + j), tab.at(tv.p3 + H + j), psi[int64_t(H + j) * a.stride],
                  psi[int64_t(H - 1 - j) * a.stride]);
        s_part[0][warp][lane] = g.s01.x;
        s_part[1][warp][lane] = g.s01.y;
        s_part[2][warp][lane] = g.s11.x;
        s_part[3][warp][lane] = g.s11.y;
        s_part[4][warp][lane] = g.s2;
        s_part[5][warp][lane] = g.s3;
    }
    __syncthreads();
    const int ngroups = (H + s.gpairs - 1) / s.gpairs;
    // each of the seven sums over the groups in a warp of its own
    if (warp < 7) {
        double acc = 0.0;
        for (int g = 0; g < ngroups; ++g) {
            const double s0 = s_part[0][g][lane], r0 = s_part[1][g][lane], s1 = s_part[2][g][lane];
            const double r1 = s_part[3][g][lane], s2 = s_part[4][g][lane], s3 = s_part[5][g][lane];
            acc += warp == 0 ? s0 : warp == 1 ? s1 : warp == 2 ? s2 + r0 : warp == 3 ? s2 : warp == 4 ? s3 : warp == 5 ? r0 : r1;
        }
        s_sum[warp][lane] = acc;
    }
    __syncthreads();
    if (warp == 0) {
        MomentSums<double> ms;
        ms.F0 = as_ff(s_sum[0][lane]);
        ms.F1 = as_ff(s_sum[1][lane]);
        ms.FE = as_ff(s_sum[2][lane]);
        ms.tS2 = s_sum[3][lane];
        ms.tS3 = s_sum[4][lane];
        ms.tR0 = s_sum[5][lane];
        ms.tR1 = s_sum[6][lane];
        double n, u, T, q;
        ms.finish(false, n, u, T, q);
        if (i >= 0 && i < a.nx && nonphysical_(n, u, T, q)) atomicOr(a.err, 1u);
        s_n[lane] = n;
        s_u[lane] = u;
        s_T[lane] = T;
        s_q[lane] = q;
    }
    __syncthreads();
    if (warp == 4 || warp == 5) {
        // Hermite coefficients of the equilibrium (Eq. g_alpha), as the tile kernels
        // hold them: warp 5 forms the recurrence's factors, kChunk orders at a time in
        // two buffers, warp 4 runs it (two instructions on its chain per order)
        const double u = s_u[lane], Tm1 = s_T[lane] - double(1);
        V *ch = static_cast<V *>(s.ch) + (i - s.i0);
        double cm2 = double(1), cm1 = u;
        if (warp == 4 && own) ch[0] = mk2(cm2, cm1);
        int buf = 0;
        for (int l0 = 2; l0 < s.Q; l0 += kChunk, buf ^= 1) {
            const int l1 = min(s.Q, l0 + kChunk);
            if (warp == 5)
#pragma unroll 8
                for (int l = l0; l < l1; ++l) {
                    if (LQ) s_fac[1][buf][l - l0][lane] = tab.at(tv.ca + l) * u;
                    s_fac[0][buf][l - l0][lane] = tab.at(tv.cb + l) * Tm1;
                }
            asm volatile("bar.sync 2, 64;" ::: "memory");  // warps 4 and 5
            if (warp == 4)
#pragma unroll 4
                for (int l = l0; l < l1; l += 2) {
                    const int r = l - l0;
                    const double ce = fma_(LQ ? s_fac[1][buf][r][lane] : u, cm1, s_fac[0][buf][r][lane] * cm2);
                    const double co = fma_(LQ ? s_fac[1][buf][r + 1][lane] : u, ce, s_fac[0][buf][r + 1][lane] * cm1);
                    if (own) ch[int64_t(l / 2) * s.cs] = mk2(ce, co);
                    cm2 = ce;
                    cm1 = co;
                }
        }
        return;
    }
    if (warp > 5) return;
    if (warp == 1) s_lnn[lane] = log_(s_n[lane]);
    if (warp == 2) s_lnT[lane] = log_(s_T[lane]);
    if (RET && warp == 3) {
        double nbar = double(1);
        if (inball) {
            // densities as fm_density (fdlb_aux.cuh): interior or periodic image, else the fixed ghosts'
            double dn = s_n[lane];
            if (!a.periodic && i < 0) dn = double(s.ghost[i < -3 ? 0 : int(i) + 3]);
            if (!a.periodic && i >= a.nx) dn = double(s.ghost[3 + int(i - a.nx > 2 ? 2 : i - a.nx)]);
            double acc = double(0);
            for (int d = 0; d <= 2 * s.W; ++d)
                acc = fma_(double(s.K[d]), __shfl_sync(0xffffffffu, dn, min(max(lane - s.W + d, 0), 31)), acc);
            nbar = acc;
        } else {
            nbar = static_cast<const double *>(a.nbar)[kHalo + source_cell_(i, a.nx, false)];
        }
        const double chi = chi_of_nbar_(a, nbar);
        s_chi[lane] = chi;
        s_lnchi[lane] = log_(chi);
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");  // warps 0 - 3
    if (warp == 0 && own) {
        const double inv_dx = double(a.inv_dx);
        const double dlnn = cd6_(s_lnn, lane) * inv_dx, du = cd6_(s_u, lane) * inv_dx, dlnT = cd6_(s_lnT, lane) * inv_dx;
        const CellCoefs<double> c =
            cell_coefs_<double, RET>(a, s.stage, s_n[lane], s_u[lane], s_T[lane], s_q[lane], dlnn, du, dlnT,
                                   RET ? s_chi[lane] : double(0), RET ? cd6_(s_lnchi, lane) * inv_dx : double(0));
        V *D = static_cast<V *>(s.coef) + (i - s.i0);
        D[0] = c.D0;
        D[s.cs] = c.D1;
        D[2 * s.cs] = c.D2;
        D[3 * s.cs] = c.D3;
        D[4 * s.cs] = sp2(c.kpsi);
    }
}

// Warp w of block (b, y): velocity pair y kPairWarps + w of cells 31 b .. 31 b + 30;
// lane l takes cell 31 b + l - 1, lane 0 the face left of the strip only.
template <int STAGE, bool LQ>
__global__ void __launch_bounds__(32 * kPairWarps) fdlb_pair_kernel(CellArgs s)
{
    using V = double2;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const StageArgs &a = s.a;
    const int lane = threadIdx.x & 31, H = s.Q / 2, j = int(blockIdx.y) * kPairWarps + (threadIdx.x >> 5);
    if (j >= H) return;
    const SetTables<LQ> tab(s);
    const TabView tv = tab.tv;
    const int64_t i = s.i0 + int64_t(blockIdx.x) * kPairCells + lane - 1;  // i0 - 1 .. nx + 30: inside the rows' columns
    const bool owner = lane != 0 && i < s.i1;
    const int64_t ic = (i < s.i0 ? s.i0 : (i < s.i1 ? i : s.i1 - 1)) - s.i0;  // lanes without a cell read another's
    const int64_t ip = int64_t(H + j) * a.stride + kHalo + i, im = int64_t(H - 1 - j) * a.stride + kHalo + i;
    const V *__restrict__ rp = static_cast<const V *>(a.in) + ip;
    const V *__restrict__ rm = static_cast<const V *>(a.in) + im;
    V bp = sp2(double(0)), bm = sp2(double(0));
    if (STAGE >= 2) {
        bp = static_cast<const V *>(a.base)[ip];
        bm = static_cast<const V *>(a.base)[im];
    }
    const V *__restrict__ D = static_cast<const V *>(s.coef) + ic;
    const V *__restrict__ ch = static_cast<const V *>(s.ch) + ic;
    // the two faces in a loop of their own body: each warp runs this code once, and
    // both side by side are twice the instructions to fetch
    V hp, hm, fp0, fm0;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        const V *r = side ? rm + 1 : rp;  // upwind stencil for +p, its mirror image for -p
        const int d = side ? -1 : 1;
        const V f0 = r[0];
        const V m2 = r[-2 * d], m1 = r[-d], p1 = r[d], p2 = r[2 * d];
        const V wa = sub2(m2, m1), wb = sub2(f0, m1), wg = sub2(p1, f0), wc = sub2(p2, p1);
        double hh[2];
        weno5_faces_i64<2>({wa.x, wa.y}, {wb.x, wb.y}, {wg.x, wg.y}, {wc.x, wc.y}, {f0.x, f0.y}, hh);
        const V h = mk2(hh[0], hh[1]);
        if (side) {
            hm = h;
            fm0 = r[-1];
        } else {
            hp = h;
            fp0 = f0;
        }
    }
    const V hpl = mk2(__shfl_up_sync(0xffffffffu, hp.x, 1), __shfl_up_sync(0xffffffffu, hp.y, 1));
    const V hml = mk2(__shfl_up_sync(0xffffffffu, hm.x, 1), __shfl_up_sync(0xffffffffu, hm.y, 1));
    // g at +p and -p: even and odd Hermite parts, the coefficients loaded kBatch ahead of the sum
    V eo = sp2(double(0));
    const int G = tv.G + (H + j) * s.Q;
    constexpr int kBatch = LQ ? 8 : 4;
    V cb[kBatch], gb[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
        cb[u] = ch[int64_t(min(u, H - 1)) * s.cs];
        gb[u] = tab.pair(G + 2 * min(u, H - 1));
    }
    for (int m = 0; m < H; m += kBatch) {
        V nc[kBatch], ng[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int at = min(m + kBatch + u, H - 1);
            nc[u] = ch[int64_t(at) * s.cs];
            ng[u] = tab.pair(G + 2 * at);
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (m + u < H) eo = fma2(gb[u], cb[u], eo);
            cb[u] = nc[u];
            gb[u] = ng[u];
        }
    }
    const double p = tab.at(tv.p + H + j), gpv = eo.x + eo.y, gmv = eo.x - eo.y;
    const V padv = sp2(p * advection_<double>(a, STAGE)), kpsi = D[4 * s.cs];
    const V E = fma2(D[2 * s.cs], sp2(tab.at(tv.p2 + H + j)), D[0]);
    const V O = mul2(fma2(D[3 * s.cs], sp2(tab.at(tv.p2 + H + j)), D[s.cs]), sp2(p));
    const V Pp = add2(E, O), Pm = sub2(E, O);
    V vp = fma2(padv, sub2(hpl, hp), fma2(fp0, kpsi, mul2(sp2(gpv), Pp)));
    V vm = fma2(padv, sub2(hm, hml), fma2(fm0, kpsi, mul2(sp2(gmv), Pm)));
    if (!owner) return;
    if (STAGE >= 2) {
        const V c = sp2(double(1) - rk_weight_<double>(STAGE));
        vp = fma2(c, bp, vp);
        vm = fma2(c, bm, vm);
    }
    V *op = static_cast<V *>(a.out) + ip, *om = static_cast<V *>(a.out) + im;
    *op = vp;
    *om = vm;
    if (STAGE != 0 && a.periodic) {  // periodic images in the ghost columns
        if (i < kHalo) {
            op[a.nx] = vp;
            om[a.nx] = vm;
        }
        if (i >= a.nx - kHalo) {
            op[-a.nx] = vp;
            om[-a.nx] = vm;
        }
    }
}

template <typename K>
static cudaError_t launch_pdl(K k, dim3 grid, dim3 block, cudaStream_t st, const CellArgs &s)
{
    // programmatic stream serialisation, as for the stage kernels
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, s);
}

// The stage of cells i0 .. i1 - 1.
template <bool LQ>
static cudaError_t cell_chunk(const CellArgs &s, bool ret, cudaStream_t st)
{
    const int64_t n = s.i1 - s.i0;
    const int halo = 3 + (ret && s.W <= kCellBall ? s.W : 0), ncell = 32 - 2 * halo;
    const dim3 cgrid(unsigned((n + ncell - 1) / ncell)), cblock(32 * kCellWarps);
    cudaError_t e = ret ? launch_pdl(fdlb_cell_kernel<true, LQ>, cgrid, cblock, st, s)
                        : launch_pdl(fdlb_cell_kernel<false, LQ>, cgrid, cblock, st, s);
    if (e != cudaSuccess) return e;
    const dim3 grid(unsigned((n + kPairCells - 1) / kPairCells), unsigned((s.Q / 2 + kPairWarps - 1) / kPairWarps));
    const dim3 block(32 * kPairWarps);
    switch (s.stage) {
    case 0: return launch_pdl(fdlb_pair_kernel<0, LQ>, grid, block, st, s);
    case 1: return launch_pdl(fdlb_pair_kernel<1, LQ>, grid, block, st, s);
    case 2: return launch_pdl(fdlb_pair_kernel<2, LQ>, grid, block, st, s);
    case 3: return launch_pdl(fdlb_pair_kernel<3, LQ>, grid, block, st, s);
    }
    return cudaErrorInvalidValue;
}

// One stage in chunks of s.cs cells, which share the per-cell buffers.
template <bool LQ>
static cudaError_t cell_stage(CellArgs s, bool ret, cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    for (s.i0 = 0; s.i0 < s.a.nx && e == cudaSuccess; s.i0 += s.cs) {
        s.i1 = s.i0 + s.cs < s.a.nx ? s.i0 + s.cs : s.a.nx;
        e = cell_chunk<LQ>(s, ret, st);
    }
    return e;
}

// One stage (s.stage); s.tab null: a tiled velocity set.
cudaError_t launch_cell_stage(CellArgs s, bool ret, cudaStream_t st)
{
    if (ret && s.W > kCellBall && !s.a.nbar) return cudaErrorInvalidValue;
    static_assert(kMaxQ / 2 <= kCellWarps * SumGroup<double>::pairs, "one warp per group");
    s.gpairs = s.tab ? (s.Q / 2 + kCellWarps - 1) / kCellWarps : SumGroup<double>::pairs;
    return s.tab ? cell_stage<true>(s, ret, st) : cell_stage<false>(s, ret, st);
}

}  // namespace qlbm
