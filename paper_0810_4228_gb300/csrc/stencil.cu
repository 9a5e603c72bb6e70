// Wilson stencil kernels: A = gamma5 D_w(mu) and A^dag = gamma5 D_w(-mu)
// (Sec. 1, Eq. 1.1-1.2; the adjoint enters the two-sided Lanczos recurrence of
// Sec. 4, Eq. 4.2), plus the layout conversions at the library boundary.
//
// One thread per lattice site, 128-thread blocks held to 80 registers so that six
// blocks (24 warps) share an SM: the single application is bound by HBM and its
// DRAM traffic is already the algorithmic minimum (links and x read once, y
// written once), so what remains is keeping enough loads in flight.  A block covers a range of checkerboard
// indices for both parities (first half of the block parity 0, second half
// parity 1), so neighbouring sites -- which have the opposite parity -- are
// processed by the same block and their links/spinors are re-read from L1/L2.
// Spinors are stored [component-chunk][site] with 16-byte chunks (double2 for
// FP64, float4 = two complex for FP32): every load of a warp is one 512-byte
// coalesced transaction.  Links are stored [nu][element][site]; the FP32 12-real
// format keeps rows 0 and 1 and rebuilds row 2 = conj(row0 x row1) in registers.
// The e^{+-mu} factors, kappa and the antiperiodic time phase are applied as
// real scalars to the projected half spinor, so links stay in SU(3).
#include <algorithm>
#include <type_traits>

#include "hop64.cuh"
#include "stencil_impl.cuh"

namespace ovl {

__device__ __forceinline__ int site_of_block(const Geom& g, int block) {
    const int half = blockDim.x >> 1;
    const int par = threadIdx.x >= half;
    const int cb = block * half + (threadIdx.x - par * half);
    return cb < g.Vh ? par * g.Vh + cb : -1;
}
__device__ __forceinline__ int site_of_thread(const Geom& g) { return site_of_block(g, blockIdx.x); }

int dslash_grid(const Geom& g, int threads) { return (g.Vh + threads / 2 - 1) / (threads / 2); }

// Row-grouped traversal of the single stencil on large lattices.  With blocks taken in index order
// the sites of hyperplane x0 + 1 come a whole hyperplane (L1 L2 L4 sites, 42 MB of spinors and
// links on 48^3 x 64) after those of x0, and the x0 neighbours and backward links fall out of L2 in
// between and are read from DRAM again (ncu: 1.45 x the algorithmic bytes there, 1.06 x on
// 32^3 x 64).  This grid visits the rows (x0, x1) as: for each group of gx consecutive x1, for
// each x0, the group's rows; blockIdx.x is the block within its row, blockIdx.y the x1 within its
// group, blockIdx.z = group * L0 + x0 (blocks are issued in linear block order: x, then y, then z).
// The x0 neighbours are then gx rows back (7 MB at gx = 8 on 48^3 x 64) and only the rows at a
// group's edges re-read an x1 neighbour.  Each site is still computed by exactly one thread, with
// the same arithmetic: the result is the same to the bit.
struct RowGrid {
    bool ok;
    dim3 grid;
};
static RowGrid row_grid(const Geom& g, int threads) {
    const int half = threads / 2;
    const int row = g.L[2] * g.L4h;  // sites of one parity in a row (x0, x1)
    if (row % half) return {false, dim3(1)};
    int gx = 1;
    for (int d = 1; d <= 16; ++d)
        if (g.L[1] % d == 0) gx = d;
    const long long z = (long long)(g.L[1] / gx) * g.L[0];
    if (z > 65535) return {false, dim3(1)};
    return {true, dim3(row / half, gx, (unsigned)z)};
}

// block bx of nx within its row
__device__ __forceinline__ int site_of_rows(const Geom& g, int bx, int nx) {
    const int half = blockDim.x >> 1;
    const int par = threadIdx.x >= half;
    const int x0 = blockIdx.z % g.L[0];
    const int x1 = (blockIdx.z / g.L[0]) * gridDim.y + blockIdx.y;
    const int cb = ((x0 * g.L[1] + x1) * nx + bx) * half + (threadIdx.x - par * half);
    return par * g.Vh + cb;
}
__device__ __forceinline__ int site_of_thread_rows(const Geom& g) {
    return site_of_rows(g, blockIdx.x, gridDim.x);
}

// --------------------------------------------- direction-split variants --
// For lattices too small to fill the GPU with one thread per site, the four
// directions of a site go to four warps of the same block (warp w computes the
// forward and backward hop of direction w for 32 consecutive sites, so no warp
// diverges); the four partial spinors meet in shared memory, and the 128
// threads then finish (site, spin) pairs: diagonal term, gamma5, scaling and
// the fused epilogue.  Four times the threads, a quarter of the dependent
// loads per thread.
static constexpr int DS_SITES = 32;

// partial spinors of the four directions: smem[dir][input][site][12]
template <int LF, int NIN>
__device__ __forceinline__ void dir_partials(const Geom& g, const void* U,
                                             const typename VecT<typename LinkReal<LF>::R>::T* const (&x)[NIN],
                                             const HopCoef<typename LinkReal<LF>::R> (&hc)[NIN],
                                             cx<typename LinkReal<LF>::R>* sm) {
    using R = typename LinkReal<LF>::R;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * DS_SITES + lane;
    Spinor<R> acc[NIN];
#pragma unroll
    for (int n = 0; n < NIN; ++n)
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int a = 0; a < 3; ++a) acc[n].s[s][a] = mk(R(0), R(0));
    if (i < g.V) {
        const Coord c = site_coord(g, i);
        switch (w) {  // uniform per warp
            case 0: hops_dir<0, LF, R, NIN>(g, c, i, U, x, acc, hc); break;
            case 1: hops_dir<1, LF, R, NIN>(g, c, i, U, x, acc, hc); break;
            case 2: hops_dir<2, LF, R, NIN>(g, c, i, U, x, acc, hc); break;
            default: hops_dir<3, LF, R, NIN>(g, c, i, U, x, acc, hc); break;
        }
    }
#pragma unroll
    for (int n = 0; n < NIN; ++n)
#pragma unroll
        for (int q = 0; q < 12; ++q) sm[((w * NIN + n) * DS_SITES + lane) * 12 + q] = acc[n].s[q / 3][q % 3];
    __syncthreads();
}

// sum of the four direction partials for (site, spin) of this thread, input n
template <class R, int NIN>
__device__ __forceinline__ void dir_sum(const cx<R>* sm, int n, int site, int sp, cx<R> (&o)[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cx<R> z = mk(R(0), R(0));
#pragma unroll
        for (int w = 0; w < 4; ++w) z = z + sm[((w * NIN + n) * DS_SITES + site) * 12 + 3 * sp + a];
        o[a] = z;
    }
}

template <int LF>
__global__ void __launch_bounds__(128) k_dslash_ds(const void* __restrict__ U,
                                                  const typename VecT<typename LinkReal<LF>::R>::T* __restrict__ x,
                                                  typename VecT<typename LinkReal<LF>::R>::T* __restrict__ y,
                                                  HopCoef<typename LinkReal<LF>::R> hc, int g5, const KState* ks,
                                                  Geom g) {
    using R = typename LinkReal<LF>::R;
    extern __shared__ __align__(16) unsigned char smraw[];
    cx<R>* sm = reinterpret_cast<cx<R>*>(smraw);
    if (ks && (ks->done || ks->status)) return;
    const typename VecT<R>::T* const xs[1] = {x};
    const HopCoef<R> hcs[1] = {hc};
    dir_partials<LF, 1>(g, U, xs, hcs, sm);
    const int site = threadIdx.x >> 2, sp = threadIdx.x & 3;
    const int i = blockIdx.x * DS_SITES + site;
    if (i >= g.V) return;
    cx<R> o[3];
    dir_sum<R, 1>(sm, 0, site, sp, o);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cx<R> z = o[a] + ld_comp<R>(x, g.V, i, 3 * sp + a);
        if (g5 && sp >= 2) z = -z;
        st_comp<R>(y, g.V, i, 3 * sp + a, z);
    }
}

template <int LF>
__global__ void __launch_bounds__(128) k_dslash_pair_ds(
    const void* __restrict__ U, const typename VecT<typename LinkReal<LF>::R>::T* __restrict__ v,
    const typename VecT<typename LinkReal<LF>::R>::T* __restrict__ w,
    typename VecT<typename LinkReal<LF>::R>::T* __restrict__ t, typename VecT<typename LinkReal<LF>::R>::T* __restrict__ s,
    HopCoef<typename LinkReal<LF>::R> hv, HopCoef<typename LinkReal<LF>::R> hw, KState* ks, double2* alpha, int step,
    int klast, double* partials, unsigned int* counter, Geom g) {
    using R = typename LinkReal<LF>::R;
    extern __shared__ __align__(16) unsigned char smraw[];
    cx<R>* sm = reinterpret_cast<cx<R>*>(smraw);
    __shared__ double red[96];
    if (ks->done || ks->status) return;
    const double2 sv = ks->sv, sw = ks->sw;
    const typename VecT<R>::T* const xs[2] = {v, w};
    const HopCoef<R> hcs[2] = {hv, hw};
    dir_partials<LF, 2>(g, U, xs, hcs, sm);
    const int site = threadIdx.x >> 2, sp = threadIdx.x & 3;
    const int i = blockIdx.x * DS_SITES + site;
    double part[3] = {0.0, 0.0, 0.0};
    if (i < g.V) {
        cx<R> ov[3], ow[3];
        dir_sum<R, 2>(sm, 0, site, sp, ov);
        dir_sum<R, 2>(sm, 1, site, sp, ow);
        const cx<R> csv = mk(R(sv.x), R(sv.y)), csw = mk(R(sw.x), R(sw.y));
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int q = 3 * sp + a;
            const cx<R> wq = ld_comp<R>(w, g.V, i, q);
            cx<R> tv = ov[a] + ld_comp<R>(v, g.V, i, q);
            cx<R> sq = ow[a] + wq;
            if (sp >= 2) {
                tv = -tv;
                sq = -sq;
            }
            tv = csv * tv;
            sq = csw * sq;
            st_comp<R>(t, g.V, i, q, tv);
            st_comp<R>(s, g.V, i, q, sq);
            const cx<double> z = cdot(up(wq), up(tv));
            part[0] += z.r;
            part[1] += z.i;
            part[2] += norm2(up(tv));
        }
    }
    double out[3];
    if (grid_sum_last<3>(part, partials, counter, out, red)) {
        if (threadIdx.x == 0) {
            const cx<double> a = cdot(d2c(sw), mk(out[0], out[1]));
            alpha[step] = c2d(a);
            const double tn = sqrt(out[2]);
            if (tn > ks->anorm) ks->anorm = tn;
            ks->kused = step + 1;
            if (step == klast) ks->done = 1;
        }
    }
}

__global__ void __launch_bounds__(128) k_dslash_regen_ds(const double2* __restrict__ U, const double2* __restrict__ vi,
                                                         const double2* __restrict__ vim1, double2* __restrict__ vip1,
                                                         double2* __restrict__ y, HopCoef<double> hc,
                                                         const KState* ks, const double2* __restrict__ alpha,
                                                         const double2* __restrict__ beta,
                                                         const double2* __restrict__ gamma,
                                                         const double2* __restrict__ c, int step, Geom g) {
    extern __shared__ __align__(16) unsigned char smraw[];
    cx<double>* sm = reinterpret_cast<cx<double>*>(smraw);
    if (ks->status || step + 1 >= ks->kused) return;
    const double2* const xs[1] = {vi};
    const HopCoef<double> hcs[1] = {hc};
    dir_partials<LINK_F64, 1>(g, U, xs, hcs, sm);
    const int site = threadIdx.x >> 2, sp = threadIdx.x & 3;
    const int i = blockIdx.x * DS_SITES + site;
    if (i >= g.V) return;
    cx<double> o[3];
    dir_sum<double, 1>(sm, 0, site, sp, o);
    const cx<double> a = d2c(alpha[step]);
    const cx<double> ib = cdiv(mk(1.0, 0.0), d2c(beta[step]));
    const cx<double> gm = step > 0 ? d2c(gamma[step - 1]) : mk(0.0, 0.0);
    const cx<double> cc = d2c(c[step + 1]);
#pragma unroll
    for (int q3 = 0; q3 < 3; ++q3) {
        const int q = 3 * sp + q3;
        const size_t e = (size_t)q * g.V + i;
        const cx<double> self = d2c(vi[e]);
        cx<double> z = o[q3] + self;
        if (sp >= 2) z = -z;
        z = z - a * self;
        if (step > 0) z = z - gm * d2c(vim1[e]);
        z = ib * z;
        vip1[e] = c2d(z);
        cx<double> yy = d2c(y[e]);
        cfma(yy, cc, z);
        y[e] = c2d(yy);
    }
}

static size_t ds_smem(int bytes_per_cx, int nin) { return (size_t)4 * nin * DS_SITES * 12 * bytes_per_cx; }
static int ds_grid(const Geom& g) { return (g.V + DS_SITES - 1) / DS_SITES; }

// one thread per site fills the GPU with the FP64 regeneration step from about this many sites up
static bool use_ds(const Geom& g) { return g.V < 152 * 1024; }

// ------------------------------------------------------------ single apply --
template <int LF, int MINB, bool ROWS>
__global__ void __launch_bounds__(128, MINB) k_dslash(const void* __restrict__ U,
                                                const typename VecT<typename LinkReal<LF>::R>::T* __restrict__ x,
                                                typename VecT<typename LinkReal<LF>::R>::T* __restrict__ y,
                                                HopCoef<typename LinkReal<LF>::R> hc, int g5, const KState* ks,
                                                Geom g) {
    using R = typename LinkReal<LF>::R;
    if (ks && (ks->done || ks->status)) return;
    const int i = ROWS ? site_of_thread_rows(g) : site_of_thread(g);
    if (i < 0) return;
    const typename VecT<R>::T* const xs[1] = {x};
    Spinor<R> acc[1];
    const HopCoef<R> hcs[1] = {hc};
    apply_site<LF, R, 1>(g, i, U, xs, acc, hcs);
    Spinor<R> self;
    load_spinor(x, g.V, i, self);
    finish_site(acc[0], self, g5 != 0);
    store_spinor(y, g.V, i, acc[0]);
}

// FP64 application with a site shared by eight lanes (RS = 1) or sixteen (RS = 2): see hop64.cuh.  CANON:
// x and y in the canonical layout ([site][12], sites in canonical order), otherwise the device layout.
// A warp takes 4 / RS consecutive sites; the half spinors meet in its own shared memory.  Bound by the FP64
// pipe: 108 FP64 instructions per four sites (RS = 1) at 19 cycles each and SM.  Measured against one thread
// per site (large lattices) and per site and direction (small ones), device layout: 4^4 15.0 -> 6.7 us,
// 24^4 695 -> 481 us.  Canonical vectors, which went through the device layout (three launches): 4^4 22.9 ->
// 6.2 us, 24^4 776 -> 481.
template <int RS, bool CANON>
__global__ void __launch_bounds__(128) k_dslash_hl(const double2* __restrict__ U, const double2* __restrict__ x,
                                                   double2* __restrict__ y, double kappa, double emu, double emum,
                                                   int g5, const KState* ks, Geom g) {
    constexpr int SPW = 4 / RS;
    __shared__ __align__(16) double2 hps[4][6 * HP_ST];
    if (ks && (ks->done || ks->status)) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int hop = lane & 7, half = RS == 2 ? (lane >> 3) & 1 : 0, sub = lane / (8 * RS);
    const int s0 = (blockIdx.x * 4 + wid) * SPW + sub;
    if (s0 - sub >= g.V) return;  // the warp's first site (uniform over the warp)
    const bool ok = s0 < g.V;
    const int s = ok ? s0 : g.V - 1;
    const size_t V = (size_t)g.V;
    int c[4];
    if (CANON) {
        int r = s;
        c[3] = r % g.L[3];
        r /= g.L[3];
        c[2] = r % g.L[2];
        r /= g.L[2];
        c[1] = r % g.L[1];
        c[0] = r / g.L[1];
    } else {
        const Coord cc = site_coord(g, s);
#pragma unroll
        for (int d = 0; d < 4; ++d) c[d] = cc.x[d];
    }
    const int nu = hop & 3;
    const bool fwd = hop < 4;
    const bool edge = nu == 3 && g.bc_t < 0 && (fwd ? c[3] == g.L[3] - 1 : c[3] == 0);
    int nc[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        int v = c[d];
        if (d == nu) {
            v += fwd ? 1 : -1;
            if (v == g.L[d]) v = 0;
            if (v < 0) v = g.L[d] - 1;
        }
        nc[d] = v;
    }
    const int ni = internal_index(g, nc);
    const int li = fwd ? (CANON ? internal_index(g, c) : s) : ni;  // the link's site
    const double2* xb = CANON ? x + (size_t)canon_index(g, nc) * 12 : x + ni;
    cx<double> o[6 / RS];
    hop_lane<RS, false>(hop, half, xb, CANON ? 1 : V, U + (size_t)nu * 9 * V + li, V, edge, o);
    double2* hp = hps[wid];
#pragma unroll
    for (int q = 0; q < 6 / RS; ++q) hp[(q + 3 * half) * HP_ST + sub * 9 + hop] = c2d(o[q]);
    const int sp = hop >> 1, part = hop & 1;
    int off[8];
    double cw[8];
    epilogue_lane(sp, part, emu, emum, off, cw);
    const unsigned sg = sp >= 2 && g5 ? SIGN : 0u;
    const double mk_ = flip(kappa, sg ^ SIGN);
    __syncwarp();
    const double* hd = reinterpret_cast<const double*>(hp + sub * 9);
    const double* xd = reinterpret_cast<const double*>(x);
    double* yd = reinterpret_cast<double*>(y);
#pragma unroll
    for (int q = 0; q < (RS == 1 ? 3 : 2); ++q) {
        const int col = RS == 1 ? q : (half ? 2 : q);
        if (RS == 2 && half && q) break;
        const size_t e = CANON ? ((size_t)s * 12 + 3 * sp + col) * 2 + part : ((3 * sp + col) * V + s) * 2 + part;
        const double z = fma(mk_, hop_sum(hd + 2 * col * HP_ST, off, cw), flip(__ldg(xd + e), sg));
        if (ok) yd[e] = z;
    }
}

template <bool CANON>
static void launch_hl(const double2* U, const double2* x, double2* y, double mu, double kappa, int gamma5,
                      const Geom& g, cudaStream_t st, const KState* ks) {
    const double ef = exp(mu), eb = exp(-mu);
    // a row of a hop per lane while that leaves at most one unit per SM quarter (4 x 152)
    if (g.V <= 2 * 608)
        k_dslash_hl<2, CANON><<<(g.V + 7) / 8, 128, 0, st>>>(U, x, y, kappa, ef, eb, gamma5, ks, g);
    else
        k_dslash_hl<1, CANON><<<(g.V + 15) / 16, 128, 0, st>>>(U, x, y, kappa, ef, eb, gamma5, ks, g);
}

void launch_dslash_canon(const double2* U, const double2* x, double2* y, double mu, double kappa, int gamma5,
                         const Geom& g, cudaStream_t st) {
    launch_hl<true>(U, x, y, mu, kappa, gamma5, g, st, nullptr);
}

// blocks per SM of the FP32 single stencil (128 threads each): 6 measured best on GB300 (48^3 x 64:
// 8 gave 4571 -> 3966 GB/s with 12-real links)
#ifndef OVL_DSLASH_F32_MINB
#define OVL_DSLASH_F32_MINB 6
#endif

static int g_ds_mode = -1;  // -1 auto, 0 one thread per site, 1 direction split
void set_dslash_variant(int mode) { g_ds_mode = mode; }
static bool pick_ds(const Geom& g) { return g_ds_mode < 0 ? use_ds(g) : g_ds_mode == 1; }

void launch_dslash(const void* U, int prec, const void* x, void* y, double mu, double kappa, int gamma5,
                   const Geom& g, cudaStream_t st, const KState* ks) {
    if (prec == 0 && g_ds_mode < 0) {
        launch_hl<false>((const double2*)U, (const double2*)x, (double2*)y, mu, kappa, gamma5, g, st, ks);
        return;
    }
    // FP32: one thread per site is the faster form from about 2^15 sites (measured, 12-real / 18-real links:
    // 20736 sites 6.4 / 6.7 us against 6.3 / 6.2 split, 36864 7.6 / 8.3 against 8.3 / 8.3, 65536 8.5 / 8.7 against
    // 10.3 / 10.4, 276480 28.5 / 32.9 against 32.9 / 45.2)
    if (g_ds_mode < 0 ? g.V < (1 << 15) : g_ds_mode == 1) {
        if (prec == 0)
            k_dslash_ds<LINK_F64><<<ds_grid(g), 128, ds_smem(16, 1), st>>>(U, (const double2*)x, (double2*)y,
                                                                          make_coef<double>(mu, kappa), gamma5, ks, g);
        else if (prec == 1)
            k_dslash_ds<LINK_F32_12><<<ds_grid(g), 128, ds_smem(8, 1), st>>>(U, (const float4*)x, (float4*)y,
                                                                            make_coef<float>(mu, kappa), gamma5, ks, g);
        else
            k_dslash_ds<LINK_F32_18><<<ds_grid(g), 128, ds_smem(8, 1), st>>>(U, (const float4*)x, (float4*)y,
                                                                            make_coef<float>(mu, kappa), gamma5, ks, g);
        return;
    }
    // FP64: four blocks per SM (128 registers; 80 spilled 1.8 KB); FP32: OVL_DSLASH_F32_MINB per SM
    const int T = 128, B = dslash_grid(g, T);
    const RowGrid rg = row_grid(g, T);
    if (prec == 0) {
        if (rg.ok)
            k_dslash<LINK_F64, 4, true><<<rg.grid, T, 0, st>>>(U, (const double2*)x, (double2*)y,
                                                                make_coef<double>(mu, kappa), gamma5, ks, g);
        else
            k_dslash<LINK_F64, 4, false><<<B, T, 0, st>>>(U, (const double2*)x, (double2*)y,
                                                           make_coef<double>(mu, kappa), gamma5, ks, g);
    } else if (prec == 1) {
        if (rg.ok)
            k_dslash<LINK_F32_12, OVL_DSLASH_F32_MINB, true><<<rg.grid, T, 0, st>>>(
                U, (const float4*)x, (float4*)y, make_coef<float>(mu, kappa), gamma5, ks, g);
        else
            k_dslash<LINK_F32_12, OVL_DSLASH_F32_MINB, false><<<B, T, 0, st>>>(
                U, (const float4*)x, (float4*)y, make_coef<float>(mu, kappa), gamma5, ks, g);
    } else {
        if (rg.ok)
            k_dslash<LINK_F32_18, OVL_DSLASH_F32_MINB, true><<<rg.grid, T, 0, st>>>(
                U, (const float4*)x, (float4*)y, make_coef<float>(mu, kappa), gamma5, ks, g);
        else
            k_dslash<LINK_F32_18, OVL_DSLASH_F32_MINB, false><<<B, T, 0, st>>>(
                U, (const float4*)x, (float4*)y, make_coef<float>(mu, kappa), gamma5, ks, g);
    }
}

// -------------------------------------------------------------- pair apply --
// t = sv * gamma5 D_w(mu) v~,  s = sw * gamma5 D_w(-mu) w~,  alpha[step] = w^dag t
// with w = sw w~.  Skipped (uniformly) once the solve is done or failed.
// The two stencils go to two sets of blocks (which = 0: t and the alpha partials; 1: s), so a thread
// carries one accumulator spinor (half the registers: more warps per SM).  which is the low bit of
// blockIdx.x, so that both find the links in L2, or with t_first (one-dimensional grids only) its upper half:
// the dearer t blocks then run first and the last wave is made of s blocks (see launch_dslash_pair).  Only the t
// blocks take part in the reduction.
// Both kinds of block run the same copy of the stencil (34 KB of instructions): with a copy each, warps of
// the two kinds on one SM waited for instructions a quarter of the time (32^4, FP32: 296 -> 230 us; 48^3 x 64:
// 1843 -> 1387 us).  Bound by issue slots and load latency, at 2.8 TB/s of its own operands.
// WIDE: FP32 data summed in FP64 (its exact products too), as the direction split does.
template <int LF, bool ROWS, bool WIDE = false>
__global__ void __launch_bounds__(128, LF == LINK_F64 ? 2 : OVL_DSLASH_F32_MINB) k_dslash_pair(const void* __restrict__ U,
                                                     const typename VecT<typename LinkReal<LF>::R>::T* __restrict__ v,
                                                     const typename VecT<typename LinkReal<LF>::R>::T* __restrict__ w,
                                                     typename VecT<typename LinkReal<LF>::R>::T* __restrict__ t,
                                                     typename VecT<typename LinkReal<LF>::R>::T* __restrict__ s,
                                                     HopCoef<typename LinkReal<LF>::R> hv,
                                                     HopCoef<typename LinkReal<LF>::R> hw, KState* ks,
                                                     double2* alpha, int step, int klast, double* partials,
                                                     unsigned int* counter, Geom g, bool t_first) {
    using R = typename LinkReal<LF>::R;
    __shared__ double red[3 * 32];  // grid_sum_last<3>: 32 doubles per value
    if (ks->done || ks->status) return;
    const double2 sv = ks->sv, sw = ks->sw;
    const unsigned nx = gridDim.x >> 1;  // blocks of each kind
    const bool halves = !ROWS && t_first;
    const int which = halves ? (int)(blockIdx.x >= nx) : (int)(blockIdx.x & 1u);
    const unsigned bx = halves ? blockIdx.x - (which ? nx : 0u) : blockIdx.x >> 1;
    const int i = ROWS ? site_of_rows(g, bx, nx) : site_of_block(g, bx);
    // per-thread sums: FP64 for FP64 data and with WIDE; otherwise exact FP32 products summed as compensated
    // FP32 pairs (TwoSum) on the FP32 pipe, widened to FP64 for the block and grid sums
    using A = typename std::conditional<sizeof(R) == 4 && !WIDE, AccF, AccD>::type;
    A pa[3];
    if (i >= 0) {  // t = sv A v~, partials of w~^dag t and |t|^2; or s = sw A^dag w~
        const typename VecT<R>::T* const xs[1] = {which ? w : v};
        Spinor<R> acc[1], self;
        HopCoef<R> hcs[1] = {hv};
        hcs[0].f[3] = which ? hw.f[3] : hv.f[3];
        hcs[0].b[3] = which ? hw.b[3] : hv.b[3];
        apply_site<LF, R, 1>(g, i, U, xs, acc, hcs);
        load_spinor(xs[0], g.V, i, self);
        finish_site(acc[0], self, true);
        const cx<R> cs = which ? mk(R(sw.x), R(sw.y)) : mk(R(sv.x), R(sv.y));
#pragma unroll
        for (int sp = 0; sp < 4; ++sp)
#pragma unroll
            for (int a = 0; a < 3; ++a) acc[0].s[sp][a] = cs * acc[0].s[sp][a];
        store_spinor(which ? s : t, g.V, i, acc[0]);
        if (!which) {
            load_spinor(w, g.V, i, self);
#pragma unroll
            for (int sp = 0; sp < 4; ++sp)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if constexpr (WIDE) {
                        acc_cdot(pa, up(self.s[sp][a]), up(acc[0].s[sp][a]));
                        acc_norm2(pa[2], up(acc[0].s[sp][a]));
                    } else {
                        acc_cdot(pa, self.s[sp][a], acc[0].s[sp][a]);  // w~^dag t
                        acc_norm2(pa[2], acc[0].s[sp][a]);
                    }
                }
        }
    }
    if (which) return;
    double part[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        if constexpr (sizeof(R) == 4 && !WIDE) part[j] = (double)pa[j].hi + (double)pa[j].lo;
        else part[j] = pa[j].v;
    }
    double out[3];
    const unsigned blk = ROWS ? bx + nx * (blockIdx.y + gridDim.y * blockIdx.z) : bx;
    const unsigned nblk = ROWS ? nx * gridDim.y * gridDim.z : nx;
    if (grid_sum_last<3>(part, partials, counter, out, red, blk, nblk)) {
        if (threadIdx.x == 0) {
            // alpha = w^dag t = conj(sw) * (w~^dag t)
            cx<double> a = cdot(d2c(sw), mk(out[0], out[1]));
            alpha[step] = c2d(a);
            const double tn = sqrt(out[2]);
            if (tn > ks->anorm) ks->anorm = tn;
            ks->kused = step + 1;
            if (step == klast) ks->done = 1;
        }
    }
}

// The pair's two stencils run in one launch, so one thread per site and stencil is the faster form from few
// sites on (us of the call, FP32 / FP64, against the direction split: 4096 sites 30.6 / 66.7 against 31.0 / 48.2,
// 8748 40.3 / 67.7 against 42.2 / 67.7, 20736 50.2 / 130 against 57.6 / 131, 65536 68.2 / 270 against 88.7 / 308, 116280 76.4
// against 125.0 in FP32).  Both forms sum alpha and |t|^2 in FP64 there (WIDE): in compensated FP32 pairs the call took
// 38.1, 38.8, 49.4 and 63.0 us, but alpha's error rose from 1e-18 to 1e-17 of the terms' magnitudes, and products of
// small or large vectors left the FP32 range.
static bool pair_ds(const Geom& g) { return g_ds_mode < 0 ? g.V < (1 << 13) : g_ds_mode == 1; }
// The allocation-free call answers for its grid (ovl_apply_pair_noalloc_blocks) and keeps the one it had.
int dslash_pair_blocks(const Geom& g) { return pick_ds(g) ? ds_grid(g) : dslash_grid(g, 128); }

void launch_dslash_pair(const void* U, int prec, const void* v, const void* w, void* t, void* s, double mu,
                        double kappa, KState* ks, double2* alpha, int step, int klast, double* partials,
                        unsigned int* counter, const Geom& g, cudaStream_t st, bool fixed_grid) {
    const bool split = fixed_grid ? pick_ds(g) : pair_ds(g);
    const int B = split ? ds_grid(g) : dslash_grid(g, 128);  // the partial-sum slots the fused reduction writes
    if (split) {
        static unsigned long long attr_dev = 0;
        if (first_use_on_device(attr_dev))
            cudaFuncSetAttribute(k_dslash_pair_ds<LINK_F64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)ds_smem(16, 2));
        if (prec == 0)
            k_dslash_pair_ds<LINK_F64><<<B, 128, ds_smem(16, 2), st>>>(
                U, (const double2*)v, (const double2*)w, (double2*)t, (double2*)s, make_coef<double>(mu, kappa),
                make_coef<double>(-mu, kappa), ks, alpha, step, klast, partials, counter, g);
        else
            k_dslash_pair_ds<LINK_F32_12><<<B, 128, ds_smem(8, 2), st>>>(
                U, (const float4*)v, (const float4*)w, (float4*)t, (float4*)s, make_coef<float>(mu, kappa),
                make_coef<float>(-mu, kappa), ks, alpha, step, klast, partials, counter, g);
        return;
    }
    // large lattices: the row-grouped block order of the single stencil (same block count, so the
    // same partial-sum slots; the partials are summed in linear block order)
    const int T = 128;
    RowGrid rg = row_grid(g, T);
    rg.grid.x *= 2;  // the two stencils
    const dim3 g1(2 * B);
    // t blocks first while the links stay in L2 (129 MB) until the s blocks come, and in FP64, which waits for its pipe
    // instead (us, interleaved / t first: FP32 20736 sites 52.3 / 52.1, 43680 64.8 / 54.1, 116280 89.0 / 76.4, 166320 78.2 / 66.0,
    // 317952 104.4 / 102.2, 706440 178.4 / 176.9, 1079296 243.8 / 250.6; FP64 43680 207 / 199, 1079296 3720 / 3700)
    const bool t_first = prec == 0 || (size_t)g.V * 192 <= (size_t)129 << 20;
    if (prec == 0) {
        if (rg.ok)
            k_dslash_pair<LINK_F64, true><<<rg.grid, T, 0, st>>>(
                U, (const double2*)v, (const double2*)w, (double2*)t, (double2*)s, make_coef<double>(mu, kappa),
                make_coef<double>(-mu, kappa), ks, alpha, step, klast, partials, counter, g,
                t_first);
        else
            k_dslash_pair<LINK_F64, false><<<g1, T, 0, st>>>(
                U, (const double2*)v, (const double2*)w, (double2*)t, (double2*)s, make_coef<double>(mu, kappa),
                make_coef<double>(-mu, kappa), ks, alpha, step, klast, partials, counter, g,
                t_first);
    } else {
        const bool wide = use_ds(g);  // up to the volume where the other forms of the call sum in FP64 (pair_ds)
        auto go = [&](auto kern, dim3 grid) {
            kern<<<grid, T, 0, st>>>(U, (const float4*)v, (const float4*)w, (float4*)t, (float4*)s,
                                     make_coef<float>(mu, kappa), make_coef<float>(-mu, kappa), ks, alpha, step, klast,
                                     partials, counter, g, t_first);
        };
        if (rg.ok)
            go(wide ? k_dslash_pair<LINK_F32_12, true, true> : k_dslash_pair<LINK_F32_12, true>, rg.grid);
        else
            go(wide ? k_dslash_pair<LINK_F32_12, false, true> : k_dslash_pair<LINK_F32_12, false>, g1);
    }
}

// ------------------------------------------------------ two-pass regeneration --
// v_{i+1} = ((A - alpha_i) v_i - gamma_{i-1} v_{i-1}) / beta_i ;  y += c_{i+1} v_{i+1}
__global__ void __launch_bounds__(256) k_dslash_regen(const double2* __restrict__ U, const double2* __restrict__ vi,
                                                      const double2* __restrict__ vim1, double2* __restrict__ vip1,
                                                      double2* __restrict__ y, HopCoef<double> hc, const KState* ks,
                                                      const double2* __restrict__ alpha,
                                                      const double2* __restrict__ beta,
                                                      const double2* __restrict__ gamma,
                                                      const double2* __restrict__ c, int step, Geom g) {
    if (ks->status || step + 1 >= ks->kused) return;
    const int i = site_of_thread(g);
    if (i < 0) return;
    const double2* const xs[1] = {vi};
    Spinor<double> acc[1];
    const HopCoef<double> hcs[1] = {hc};
    apply_site<LINK_F64, double, 1>(g, i, U, xs, acc, hcs);
    Spinor<double> self;
    load_spinor(vi, g.V, i, self);
    finish_site(acc[0], self, true);
    const cx<double> a = d2c(alpha[step]);
    const cx<double> ib = cdiv(mk(1.0, 0.0), d2c(beta[step]));
    const cx<double> gm = step > 0 ? d2c(gamma[step - 1]) : mk(0.0, 0.0);
    const cx<double> cc = d2c(c[step + 1]);
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const size_t e = (size_t)(3 * sp + q) * g.V + i;
            cx<double> z = acc[0].s[sp][q] - a * self.s[sp][q];
            if (step > 0) z = z - gm * d2c(vim1[e]);
            z = ib * z;
            vip1[e] = c2d(z);
            cx<double> yy = d2c(y[e]);
            cfma(yy, cc, z);
            y[e] = c2d(yy);
        }
}

void launch_dslash_regen(const double2* U, const double2* vi, const double2* vim1, double2* vip1, double2* y,
                         double mu, double kappa, const KState* ks, const double2* alpha, const double2* beta,
                         const double2* gamma, const double2* c, int step, const Geom& g, cudaStream_t st) {
    if (pick_ds(g)) {
        k_dslash_regen_ds<<<ds_grid(g), 128, ds_smem(16, 1), st>>>(U, vi, vim1, vip1, y, make_coef<double>(mu, kappa),
                                                                   ks, alpha, beta, gamma, c, step, g);
        return;
    }
    const int T = 128, B = dslash_grid(g, T);
    k_dslash_regen<<<B, T, 0, st>>>(U, vi, vim1, vip1, y, make_coef<double>(mu, kappa), ks, alpha, beta, gamma, c,
                                    step, g);
}

// FP64 device-layout vectors (double2 [12][V]) to the FP32 device layout (float4 [6][V],
// components 2c, 2c+1 in one float4): nvec consecutive vectors of 12V complex each.
__global__ void k_native_f64_to_f32(const double2* __restrict__ x, float4* __restrict__ y, int V, int nvec) {
    const size_t tot = (size_t)nvec * 6 * V;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x) {
        const size_t vec = e / ((size_t)6 * V);
        const size_t r = e - vec * 6 * V;
        const int c2 = (int)(r / V), i = (int)(r - (size_t)c2 * V);
        const double2* xv = x + vec * 12 * (size_t)V;
        const double2 a = xv[(size_t)(2 * c2) * V + i], b = xv[(size_t)(2 * c2 + 1) * V + i];
        y[vec * 6 * (size_t)V + (size_t)c2 * V + i] = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
    }
}

void launch_native_f64_to_f32(const double2* x, void* y, const Geom& g, int nvec, cudaStream_t st) {
    const size_t tot = (size_t)nvec * 6 * g.V;
    int blocks = (int)std::min<size_t>((tot + 255) / 256, 4096);
    k_native_f64_to_f32<<<blocks, 256, 0, st>>>(x, (float4*)y, g.V, nvec);
}

// the inverse: FP32 device layout (float4 [6][V]) to the FP64 device layout (double2 [12][V])
__global__ void k_native_f32_to_f64(const float4* __restrict__ x, double2* __restrict__ y, int V, int nvec) {
    const size_t tot = (size_t)nvec * 6 * V;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x) {
        const size_t vec = e / ((size_t)6 * V);
        const size_t r = e - vec * 6 * V;
        const int c2 = (int)(r / V), i = (int)(r - (size_t)c2 * V);
        const float4 a = x[vec * 6 * (size_t)V + (size_t)c2 * V + i];
        double2* yv = y + vec * 12 * (size_t)V;
        yv[(size_t)(2 * c2) * V + i] = make_double2((double)a.x, (double)a.y);
        yv[(size_t)(2 * c2 + 1) * V + i] = make_double2((double)a.z, (double)a.w);
    }
}

void launch_native_f32_to_f64(const void* x, double2* y, const Geom& g, int nvec, cudaStream_t st) {
    const size_t tot = (size_t)nvec * 6 * g.V;
    int blocks = (int)std::min<size_t>((tot + 255) / 256, 4096);
    k_native_f32_to_f64<<<blocks, 256, 0, st>>>((const float4*)x, y, g.V, nvec);
}

// Neighbour table: nbr[h][i] = internal index of the neighbour of site i in hop h (h < 4: x + nu,
// h >= 4: x - nu, nu = h & 3), bit-inverted (~index, negative) where the hop crosses the
// antiperiodic time boundary and takes the phase -1.
__global__ void k_build_nbr(int* __restrict__ nbr, Geom g) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.V) return;
    const Coord c = site_coord(g, i);
    for (int h = 0; h < 8; ++h) {
        const int nu = h & 3;
        const bool fwd = h < 4;
        const int nb = neighbour(g, c, nu, fwd ? +1 : -1);
        const bool edge = nu == 3 && (fwd ? (c.x[3] == g.L[3] - 1) : (c.x[3] == 0));
        nbr[(size_t)h * g.V + i] = (edge && g.bc_t < 0) ? ~nb : nb;
    }
}

void launch_build_nbr(int* nbr, const Geom& g, cudaStream_t st) {
    k_build_nbr<<<(g.V + 127) / 128, 128, 0, st>>>(nbr, g);
}

// ---------------------------------------------------------------- layouts --
// One link per thread: a block is 32 sites (device order) x 4 directions, a warp per direction, so that every
// store is one coalesced transaction and the four warps share the sites' 576-byte canonical records in L1.
// Bound by HBM (2208 bytes per site in and out).  24^4: 186 -> 177 us against one site per thread.
__global__ void __launch_bounds__(128) k_pack_gauge(const double2* __restrict__ Uc, double2* __restrict__ U64,
                                                    float4* __restrict__ U12, float2* __restrict__ U18,
                                                    float4* __restrict__ Udf, Geom g) {
    const int i = blockIdx.x * 32 + (threadIdx.x & 31), nu = threadIdx.x >> 5;
    if (i >= g.V) return;
    const Coord c = site_coord(g, i);
    const double2* u = Uc + ((size_t)canon_index(g, c.x) * 4 + nu) * 9;
    double2 e[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) e[q] = __ldg(u + q);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const size_t o = ((size_t)nu * 9 + q) * g.V + i;
        U64[o] = e[q];
        U18[o] = make_float2((float)e[q].x, (float)e[q].y);
        const dfc d = c2dfc(d2df(e[q]));
        Udf[o] = make_float4(d.rh, d.rl, d.ih, d.il);
    }
    U12[((size_t)nu * 3 + 0) * g.V + i] = make_float4(e[0].x, e[0].y, e[1].x, e[1].y);
    U12[((size_t)nu * 3 + 1) * g.V + i] = make_float4(e[2].x, e[2].y, e[3].x, e[3].y);
    U12[((size_t)nu * 3 + 2) * g.V + i] = make_float4(e[4].x, e[4].y, e[5].x, e[5].y);
}

__global__ void k_f64_to_df(void* x, size_t n) {
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const double2 v = reinterpret_cast<double2*>(x)[e];
        reinterpret_cast<dfc*>(x)[e] = c2dfc(d2df(v));
    }
}
void launch_f64_to_df(void* x, size_t n, cudaStream_t st) {
    k_f64_to_df<<<(int)std::min<size_t>((n + 255) / 256, 2048), 256, 0, st>>>(x, n);
}

void launch_pack_gauge(const double2* U_canon, double2* U64, float4* U12, float2* U18, float4* Udf, const Geom& g,
                       cudaStream_t st) {
    k_pack_gauge<<<(g.V + 31) / 32, 128, 0, st>>>(U_canon, U64, U12, U18, Udf, g);
}

__global__ void k_pack_spinor(const double2* __restrict__ canon, void* __restrict__ native, int prec, Geom g) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.V) return;
    const Coord c = site_coord(g, i);
    const int s = canon_index(g, c.x);
    if (prec == 0) {
        double2* o = (double2*)native;
        for (int q = 0; q < 12; ++q) o[(size_t)q * g.V + i] = canon[(size_t)s * 12 + q];
    } else {
        float4* o = (float4*)native;
        for (int q = 0; q < 6; ++q) {
            double2 a = canon[(size_t)s * 12 + 2 * q], b = canon[(size_t)s * 12 + 2 * q + 1];
            o[(size_t)q * g.V + i] = make_float4(a.x, a.y, b.x, b.y);
        }
    }
}

void launch_pack_spinor(const double2* canon, void* native, int prec, const Geom& g, cudaStream_t st) {
    k_pack_spinor<<<(g.V + 127) / 128, 128, 0, st>>>(canon, native, prec, g);
}

__global__ void k_unpack_spinor(const void* __restrict__ native, int prec, double2* __restrict__ canon,
                                const double2* __restrict__ b, int g5, Geom g) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.V) return;
    const Coord c = site_coord(g, i);
    const int s = canon_index(g, c.x);
    for (int q = 0; q < 12; ++q) {
        double2 v;
        if (prec == 0) {
            v = ((const double2*)native)[(size_t)q * g.V + i];
        } else {
            float4 f = ((const float4*)native)[(size_t)(q / 2) * g.V + i];
            v = (q & 1) ? make_double2(f.z, f.w) : make_double2(f.x, f.y);
        }
        if (g5 && q >= 6) v = make_double2(-v.x, -v.y);
        if (b) {
            double2 bb = b[(size_t)s * 12 + q];
            v.x += bb.x;
            v.y += bb.y;
        }
        canon[(size_t)s * 12 + q] = v;
    }
}

void launch_unpack_spinor(const void* native, int prec, double2* canon, const double2* b_canon, int g5,
                          const Geom& g, cudaStream_t st) {
    k_unpack_spinor<<<(g.V + 127) / 128, 128, 0, st>>>(native, prec, canon, b_canon, g5, g);
}

}  // namespace ovl
