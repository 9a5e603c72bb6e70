// FP64 two-sided Lanczos on lattices that fit the GPU's shared memory: all k steps (Sec. 4, Eq. 4.2) in one
// cooperative launch, and the FP64 regeneration pass of the mixed solves (Sec. 5) likewise.
//
// What bounds both is GB300's FP64 pipe.  Measured: a warp issues one FP64 instruction per 64 cycles,
// whatever its dependences and however few lanes take part, and an SM one per 19 (four warps or more).
// So every SM quarter should carry the same number of FP64 warp instructions with all lanes at work, and
// serial scalar algebra costs 64 cycles an operation (a library square root 680).  One thread per site and
// direction, the layout of the per-step kernels, left 111 of 152 SMs idle on 6^4 (41 blocks of 32 sites)
// and spent as much on butterfly sums and repeated scalar algebra as on the recurrence.
//
// Here a site is shared by 8 RS lanes per input vector: one hop each (RS = 1) or one spin row of a hop each
// (RS = 2, twice as many units of half the work, for lattices that leave SM quarters idle otherwise).  The
// hop of a lane is a runtime value: address offsets and sign-bit masks select the spin projection, the
// adjoint and the phase, so every lane runs the same instructions and none of them is an FP64 negation.
// The half spinors meet in the warp's own shared memory (no block barrier); then the same lanes take
// (spin, real or imaginary part) and sum the eight hops, signs and e^{+-mu} in the fused multiply-adds: 84 + 24 FP64 instructions per lane and unit instead of 120 + 36.  Units go round-robin
// to the blocks and then to their warps, one block per SM.  Own-site vectors stay in shared memory;
// neighbours are read through L2 (.cg), as other blocks write them.
//
// Sums: transposed warp reductions (each step halves the values a lane still carries), block partials, one
// bounded grid barrier, after which four warps of every block add all partials in the same order: all
// blocks hold identical coefficients.  The scalars of a step are formed by lanes side by side (real and
// imaginary parts, both reciprocal square roots in one instruction stream), the breakdown checks by
// another warp.
//
// Measured (GB300): FP64 solve on 6^4, k = 480, 23.0 -> 7.7 ms (48 -> 14.4 us per step, of which the FP64 pipe
// of the busiest SM quarter is busy 11); regeneration on 8^4 15.5 -> 10.5 us per step (FP64 pipe 8.5).
#include <algorithm>

#include "hop64.cuh"
#include "split64.h"

namespace ovl {
namespace {

constexpr int LT = 32 * LW;
constexpr long long LSPIN = 20000000;  // polls before a barrier wait gives up (sets ks->timeout)

// Sums over the lanes of one input (lane bit NB = 8 RS): v0 and v1 each, valid in the lane of that input
// whose lower bits are 0 (v0) or 4 (v1).  First step: the lane bit above or below NB.
template <int RS>
__device__ __forceinline__ double warp_sum_pairs(double v0, double v1) {
    constexpr int X = RS == 1 ? 16 : 8;
    v0 += __shfl_xor_sync(0xffffffffu, v0, X);
    v1 += __shfl_xor_sync(0xffffffffu, v1, X);
    const bool up = (threadIdx.x & 4) != 0;
    const double send = up ? v0 : v1, keep = up ? v1 : v0;
    double r = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    return r;
}
// the four sums of warp_sum_pairs -> red[warp][input * 2 + value]
template <int RS>
__device__ __forceinline__ void store_pairs(double r, double (&red)[4]) {
    const int lane = threadIdx.x & 31, low = lane & ~(8 * RS);
    if (low == 0 || low == 4) red[(lane & (8 * RS) ? 2 : 0) + (low >> 2)] = r;
}

// Block sums of the four values red[warp][4] of `nw` warps -> part[4 * block ..]; one warp.
__device__ __forceinline__ void block_partials(const double (*red)[4], int nw, double* part) {
    const int lane = threadIdx.x & 31, v = lane & 3, j = lane >> 2;
    double s = j < nw ? red[j][v] : 0.0;
    if (nw > 8) s += j + 8 < nw ? red[j + 8][v] : 0.0;
    if (nw > 4) s += __shfl_xor_sync(0xffffffffu, s, 16);
    if (nw > 2) s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    if (lane < 4) part[4 * blockIdx.x + v] = s;
}

// Sums over the G blocks' partials in a fixed order: warps 0..3 (one per SM quarter) a quarter each ...
__device__ __forceinline__ void grid_partials(const double* part, int G, int wid, double (*gs)[4]) {
    const int lane = threadIdx.x & 31, v = lane & 3, j = lane >> 2;
    const int b0 = wid * 8 + j;
    double x[5];
#pragma unroll
    for (int u = 0; u < 5; ++u) x[u] = b0 + 32 * u < G ? __ldcg(part + 4 * (b0 + 32 * u) + v) : 0.0;
    double s = x[0];
#pragma unroll
    for (int u = 1; u < 5; ++u)
        if (32 * u < G) s += x[u];
    for (int b = b0 + 160; b < G; b += 32) s += __ldcg(part + 4 * b + v);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    if (lane < 4) gs[wid][v] = s;
}
// ... and, behind a block barrier, their sum in every lane of the calling warp
__device__ __forceinline__ void grid_sums(const double (*gs)[4], double (&o)[4]) {
    const int lane = threadIdx.x & 31, v = lane & 3, j = (lane >> 2) & 1;
    double s = gs[2 * j][v] + gs[2 * j + 1][v];
    s += __shfl_xor_sync(0xffffffffu, s, 4);
#pragma unroll
    for (int q = 0; q < 4; ++q) o[q] = __shfl_sync(0xffffffffu, s, q);
}

struct L2Args {
    const double2* U;
    const int* nbr;
    double2* v[3];        // ring of three, or v[0] + i * vstep when vstep > 0 (stored basis)
    double2* w[3];
    size_t vstep, wstep;
    KState* ks;
    double2 *alpha, *beta, *gamma, *vscale;
    double* partA;        // [G][4]
    double* partC;        // [G][4]
    unsigned int* bar;
    double kappa, emu, emum;
    int V, k, npass;
    long long spin;       // limit of a barrier wait's polls (LIM)
};

// shared memory: half spinors of a warp's units, then own-site state [pass][cur, prev, t][value][thread]
// (a lane holds three colours of one part of a spin, or with RS = 2 two or one of them)
constexpr int L2_HP = 6 * HP_ST;  // double2 per warp
template <int RS> constexpr int NCOL = RS == 1 ? 3 : 2;
size_t l2_smem(int rs, int npass) {
    return (size_t)LW * L2_HP * sizeof(double2) + (size_t)npass * 3 * (rs == 1 ? 3 : 2) * LT * sizeof(double);
}

// LIM: the limit of ovl_set_wait_limit in place of LSPIN.  A form of its own: with the limit an argument of the one
// form its polls, or what else the compiler then arranges otherwise, cost 0.3 to 1.6 % of a solve.
template <int RS, bool LIM>
__global__ void __launch_bounds__(LT) k_l2_f64(L2Args a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    KState* ks = a.ks;
    if (ks->done || ks->status) return;
    constexpr int NC = NCOL<RS>, NB = 8 * RS, SPW = 2 / RS;  // colours per lane, lane bit of the input, sites
    __shared__ double red[LW][4];
    __shared__ double gs[4][4];
    __shared__ double2 cs[2];   // sv, sw
    __shared__ double2 cc[4];   // alpha sv, conj(alpha) sw, gamma_{i-1} svp, conj(beta_{i-1}) swp
    __shared__ int sdone;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    double2* hp = reinterpret_cast<double2*>(smraw) + wid * L2_HP;
    double* st = reinterpret_cast<double*>(reinterpret_cast<double2*>(smraw) + LW * L2_HP) + tid;
    auto slot = [&](int p, int s, int c) -> double* { return st + ((p * 3 + s) * NC + c) * LT; };
    const int hop = lane & 7, half = RS == 2 ? (lane >> 3) & 1 : 0, n = (lane & NB) ? 1 : 0;
    const int sub = RS == 1 ? lane >> 4 : 0;   // site of the unit
    const int sp = hop >> 1, part = hop & 1;   // epilogue role of the lane; colours 0, 1 or 2 with RS = 2
    const int col0 = RS == 2 && half ? 2 : 0, ncol = RS == 1 ? 3 : 2 - half;
    const size_t V = (size_t)a.V;
    const int G = gridDim.x, nunits = a.V / SPW;
    // warps of this block that hold units
    const int nw = min(LW, (nunits - (int)blockIdx.x + G - 1) / G);
    int off[8];
    double cw[8];
    epilogue_lane(sp, part, n ? a.emum : a.emu, n ? a.emu : a.emum, off, cw);  // A^dag = gamma5 D_w(-mu)
    const int grp = (sub * 2 + n) * 9;
    const unsigned g5 = sp >= 2 ? SIGN : 0u, pneg = part ? 0u : SIGN;
    const double mk_ = flip(a.kappa, g5 ^ SIGN);
    int* err = &ks->timeout;
    for (int p = 0; p < a.npass; ++p) {
        const int u = blockIdx.x + G * (wid + LW * p);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const double* x = reinterpret_cast<const double*>(n ? a.w[0] : a.v[0]);
            const bool ok = u < nunits && c < ncol;
            *slot(p, 0, c) = ok ? x[((3 * sp + col0 + c) * V + SPW * u + sub) * 2 + part] : 0.0;
            *slot(p, 1, c) = 0.0;
        }
    }
    // recurrence scalars, in every lane of warp 0 (sv is real); what the breakdown checks need, in warp 1
    double svr = ks->sv.x, svpr = ks->svp.x, swr = ks->sw.x, swi = ks->sw.y, swpr = ks->swp.x, swpi = ks->swp.y;
    double anorm2 = ks->anorm * ks->anorm;
    int kused = 0, bd = -1;
    unsigned int nbar = 0;
    if (tid == 0) {
        cs[0] = make_double2(svr, 0.0);
        cs[1] = make_double2(swr, swi);
        cc[2] = cc[3] = make_double2(0.0, 0.0);
        sdone = 0;
    }
    __syncthreads();
    for (int i = 0; i < a.k; ++i) {
        const int cur = i & 1, prv = cur ^ 1;
        const double2* x = n ? (a.wstep ? a.w[0] + i * a.wstep : a.w[i % 3]) : (a.vstep ? a.v[0] + i * a.vstep : a.v[i % 3]);
        double* xn = reinterpret_cast<double*>(n ? (a.wstep ? a.w[0] + (i + 1) * a.wstep : a.w[(i + 1) % 3])
                                                 : (a.vstep ? a.v[0] + (i + 1) * a.vstep : a.v[(i + 1) % 3]));
        // ---- t = sv A v~_i, s = sw A^dag w~_i; partials of w~^dag t and |t|^2
        if (wid < nw) {
            double r0 = 0.0, r1 = 0.0, r2 = 0.0;
            const double sr = cs[n].x, si = flip(cs[n].y, pneg);
            for (int p = 0; p < a.npass; ++p) {
                const int u = blockIdx.x + G * (wid + LW * p);
                if (u >= nunits) break;  // uniform over the warp
                const int site = SPW * u + sub;
                cx<double> o[6 / RS];
                const int ne = __ldg(a.nbr + hop * V + site), nb = ne < 0 ? ~ne : ne;
                hop_lane<RS, true>(hop, half, x + nb, V, a.U + (size_t)(hop & 3) * 9 * V + (hop < 4 ? site : nb), V,
                                   ne < 0, o);
#pragma unroll
                for (int c = 0; c < 6 / RS; ++c) hp[(c + 3 * half) * HP_ST + grp + hop] = c2d(o[c]);
                __syncwarp();
                const double* hd = reinterpret_cast<const double*>(hp + grp);
                double z[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const int col = RS == 1 ? c : min(col0 + c, 2);
                    z[c] = fma(mk_, hop_sum(hd + 2 * col * HP_ST, off, cw), flip(*slot(p, cur, c), g5));
                }
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const double zo = __shfl_xor_sync(0xffffffffu, z[c], 1);
                    const double t = c < ncol ? fma(si, zo, sr * z[c]) : 0.0;
                    *slot(p, 2, c) = t;
                    if (n == 0) {
                        // w~ at the own site, this part and the other one: lanes of the second input
                        const double wv = slot(p, cur, c)[NB], wo = slot(p, cur, c)[part ? NB - 1 : NB + 1];
                        r0 = fma(wv, t, r0);
                        r1 = fma(flip(wo, pneg), t, r1);
                        r2 = fma(t, t, r2);
                    }
                }
                __syncwarp();  // hp is rewritten by the next pass
            }
            // the lanes of v hold (r0, r1), those of w take r2
            const double m = __shfl_xor_sync(0xffffffffu, r2, NB);
            store_pairs<RS>(warp_sum_pairs<RS>(n ? m : r0, n ? 0.0 : r1), red[wid]);
        }
        __syncthreads();
        if (wid == 0) block_partials(red, nw, a.partA);
        grid_barrier_mono(a.bar, (unsigned)G * (++nbar), err, 1, LIM ? a.spin : LSPIN);
        if (*(volatile int*)err) return;
        if (wid < 4) grid_partials(a.partA, G, wid, gs);
        __syncthreads();
        if (wid == 0) {  // alpha = conj(sw) w~^dag t: even lanes its real part, odd lanes its imaginary part
            double o[4];
            grid_sums(gs, o);
            const bool q = lane & 1;
            const double al = fma(swr, q ? o[1] : o[0], swi * (q ? flip(o[0], SIGN) : o[1]));
            const double ao = __shfl_xor_sync(0xffffffffu, al, 1);
            // lanes 0, 1: conj(alpha) sw; lanes 2, 3: alpha sv
            const double ar = q ? ao : al, ai = q ? al : ao;
            const bool first = lane < 2;
            const double m1 = first ? (q ? swi : swr) : svr, m2 = first ? (q ? flip(swr, SIGN) : swi) : 0.0;
            const double r = fma(first ? ar : al, m1, ai * m2);
            if (lane < 4) reinterpret_cast<double*>(cc)[(first ? 2 : 0) + q] = r;
            if (blockIdx.x == 0 && lane < 2) reinterpret_cast<double*>(a.alpha + i)[lane] = al;
        } else if (wid == 1) {
            double o[4];
            grid_sums(gs, o);
            anorm2 = fmax(anorm2, o[2]);
            kused = i + 1;
        }
        if (i == a.k - 1) break;
        __syncthreads();
        // ---- v^ = t - alpha v_i - gamma_{i-1} v_{i-1}, w^ likewise (Eq. 4.2)
        if (wid < nw) {
            double q0 = 0.0, q1 = 0.0;
            const double c0r = flip(cc[n].x, SIGN), c0i = flip(cc[n].y, pneg ^ SIGN);
            const double c1r = flip(cc[2 + n].x, SIGN), c1i = flip(cc[2 + n].y, pneg ^ SIGN);
            const unsigned wneg = n && part ? SIGN : 0u;
            const int po = part ? -1 : 1;
            for (int p = 0; p < a.npass; ++p) {
                const int u = blockIdx.x + G * (wid + LW * p);
                if (u >= nunits) break;
                double z[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    z[c] = fma(c0r, *slot(p, cur, c), *slot(p, 2, c));
                    z[c] = fma(c0i, slot(p, cur, c)[po], z[c]);
                    z[c] = fma(c1r, *slot(p, prv, c), z[c]);
                    z[c] = fma(c1i, slot(p, prv, c)[po], z[c]);
                }
                __syncwarp();  // the partner has read the previous vector
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    *slot(p, prv, c) = z[c];
                    if (c < ncol) xn[((3 * sp + col0 + c) * V + SPW * u + sub) * 2 + part] = z[c];
                    // lanes of v: Re += v_p w_p; lanes of w: Im += +-w_p v_{1-p}
                    const double m0 = __shfl_xor_sync(0xffffffffu, z[c], NB);
                    const double m1 = __shfl_xor_sync(0xffffffffu, m0, 1);
                    q0 = fma(flip(z[c], wneg), n ? m1 : m0, q0);
                    q1 = fma(z[c], z[c], q1);
                }
            }
            store_pairs<RS>(warp_sum_pairs<RS>(q0, q1), red[wid]);  // Re, |v^|^2, Im, |w^|^2
        }
        __syncthreads();
        if (wid == 0) block_partials(red, nw, a.partC);
        grid_barrier_mono(a.bar, (unsigned)G * (++nbar), err, 1, LIM ? a.spin : LSPIN);
        if (*(volatile int*)err) return;
        if (wid < 4) grid_partials(a.partC, G, wid, gs);
        __syncthreads();
        double nv = 0.0, gm = 0.0, rnv = 0.0, f = 0.0, dq = 0.0;
        if (wid == 0) {
            // beta = |v^|, gamma = delta / beta, sv = 1 / beta, sw = 1 / conj(gamma) = delta beta / |delta|^2
            double o[4];
            grid_sums(gs, o);
            const bool q = lane & 1;
            const double nd2 = fma(o[2], o[2], o[0] * o[0]);
            const double r = rsqrt(q ? nd2 : o[1]);         // even lanes 1 / |v^|, odd lanes 1 / |delta|
            const double r2 = r * (q ? r : o[1]);           // |v^|, 1 / |delta|^2
            rnv = __shfl_sync(0xffffffffu, r, 0);
            nv = __shfl_sync(0xffffffffu, r2, 0);
            f = nv * __shfl_sync(0xffffffffu, r2, 1);
            dq = q ? o[2] : o[0];
            gm = dq * (lane < 2 ? rnv : f);                 // lanes 0, 1: gamma; lanes 2, 3: sw
            // the next step's gamma_{i-1} svp and conj(beta_{i-1}) swp
            const double old = lane < 2 ? svr : (q ? swi : swr);
            const double cn = (lane < 2 ? gm : nv) * old;
            if (lane < 4) reinterpret_cast<double*>(cc)[4 + lane] = cn;
        } else if (wid == 1) {
            double o[4];
            grid_sums(gs, o);
            const double nd2 = fma(o[2], o[2], o[0] * o[0]);
            int dn = 0;
            if (o[1] <= 1e-26 * fmax(anorm2, 1e-300)) {
                dn = 1;  // lucky breakdown: |v^| <= 1e-13 max |A v_i|
            } else if (nd2 <= 1e-28 * o[1] * o[3]) {
                dn = 1;  // serious breakdown: |w^^dag v^| <= 1e-14 |v^| |w^|
                bd = i + 1;
            }
            if (lane == 0) sdone = dn;
        }
        __syncthreads();
        if (sdone) break;
        if (wid == 0) {
            svpr = svr, swpr = swr, swpi = swi;
            svr = rnv;
            swr = __shfl_sync(0xffffffffu, gm, 2);
            swi = __shfl_sync(0xffffffffu, gm, 3);
            if (lane == 0) {
                cs[0] = make_double2(svr, 0.0);
                cs[1] = make_double2(swr, swi);
            }
            const double gi = __shfl_sync(0xffffffffu, gm, 1);
            if (blockIdx.x == 0 && lane == 0) {
                a.beta[i] = make_double2(nv, 0.0);
                a.gamma[i] = make_double2(gm, gi);
                if (a.vscale) a.vscale[i + 1] = make_double2(svr, 0.0);
            }
        }
        __syncthreads();
    }
    if (blockIdx.x == 0 && tid == 0) {
        ks->sv = make_double2(svr, 0.0);
        ks->sw = make_double2(swr, swi);
        ks->svp = make_double2(svpr, 0.0);
        ks->swp = make_double2(swpr, swpi);
    }
    if (blockIdx.x == 0 && tid == 32) {
        ks->kused = kused;
        ks->done = 1;
        ks->anorm = sqrt(anorm2);
        if (bd >= 0) ks->bdstep = bd;
    }
}

// ---- FP64 regeneration: v_{i+1} = ((A - alpha_i) v_i - gamma_{i-1} v_{i-1}) / beta_i, y += c_{i+1} v_{i+1}
// (Sec. 5), eight lanes per site, four sites per warp, one grid barrier per step.  Coefficients per step:
// 1 / beta_i, alpha_i / beta_i, gamma_{i-1} / beta_i, c_{i+1} (k_pass2_coef).
struct R64Args {
    const double2* U;
    const int* nbr;
    double2* v[3];
    double2* y;
    const KState* ks;
    const double2* cf;  // [k][4]
    unsigned int* bar;
    int* err;
    double kappa, emu, emum;
    int V, npass;
    long long spin;       // (LIM)
};

template <int RS, bool LIM>
__global__ void __launch_bounds__(LT) k_regen_f64(R64Args a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    if (a.ks->status || a.ks->timeout) return;  // (pass 1 gave up: the same decision in every block)
    const int kused = a.ks->kused;
    constexpr int NC = NCOL<RS>, SPW = 4 / RS;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    double2* hp = reinterpret_cast<double2*>(smraw) + wid * L2_HP;
    double* st = reinterpret_cast<double*>(reinterpret_cast<double2*>(smraw) + LW * L2_HP) + tid;
    auto slot = [&](int p, int s, int c) -> double* { return st + ((p * 3 + s) * NC + c) * LT; };  // cur, prev, y
    const int hop = lane & 7, half = RS == 2 ? (lane >> 3) & 1 : 0, sub = lane / (8 * RS);
    const int sp = hop >> 1, part = hop & 1;
    const int col0 = RS == 2 && half ? 2 : 0, ncol = RS == 1 ? 3 : 2 - half;
    const size_t V = (size_t)a.V;
    const int G = gridDim.x, nunits = (a.V + SPW - 1) / SPW;
    int off[8];
    double cw[8];
    epilogue_lane(sp, part, a.emu, a.emum, off, cw);
    const int grp = sub * 9;
    const unsigned g5 = sp >= 2 ? SIGN : 0u, pneg = part ? 0u : SIGN;
    const double mk_ = flip(a.kappa, g5 ^ SIGN);
    const int po = part ? -1 : 1;
    for (int p = 0; p < a.npass; ++p) {
        const int site = SPW * (blockIdx.x + G * (wid + LW * p)) + sub;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const bool ok = site < a.V && c < ncol;
            const size_t e = ((3 * sp + col0 + c) * V + site) * 2 + part;
            *slot(p, 0, c) = ok ? reinterpret_cast<const double*>(a.v[0])[e] : 0.0;
            *slot(p, 1, c) = 0.0;
            *slot(p, 2, c) = ok ? reinterpret_cast<const double*>(a.y)[e] : 0.0;
        }
    }
    __syncwarp();
    unsigned int nbar = 0;
    for (int i = 0; i + 1 < kused; ++i) {
        const int cur = i & 1, prv = cur ^ 1;
        const double2* x = a.v[i % 3];
        double* xn = reinterpret_cast<double*>(a.v[(i + 1) % 3]);
        const double ib = __ldg(a.cf + 4 * i).x;
        const double2 ca = __ldg(a.cf + 4 * i + 1), cg = __ldg(a.cf + 4 * i + 2), cy = __ldg(a.cf + 4 * i + 3);
        const double car = flip(ca.x, SIGN), cai = flip(ca.y, pneg ^ SIGN);
        const double cgr = flip(cg.x, SIGN), cgi = flip(cg.y, pneg ^ SIGN), cyi = flip(cy.y, pneg);
        for (int p = 0; p < a.npass; ++p) {
            const int u = blockIdx.x + G * (wid + LW * p);
            if (u >= nunits) break;  // uniform over the warp
            const bool ok = SPW * u + sub < a.V;
            const int site = ok ? SPW * u + sub : a.V - 1;
            cx<double> o[6 / RS];
            const int ne = __ldg(a.nbr + hop * V + site), nb = ne < 0 ? ~ne : ne;
            hop_lane<RS, true>(hop, half, x + nb, V, a.U + (size_t)(hop & 3) * 9 * V + (hop < 4 ? site : nb), V, ne < 0,
                               o);
#pragma unroll
            for (int c = 0; c < 6 / RS; ++c) hp[(c + 3 * half) * HP_ST + grp + hop] = c2d(o[c]);
            __syncwarp();
            const double* hd = reinterpret_cast<const double*>(hp + grp);
            double z[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int col = RS == 1 ? c : min(col0 + c, 2);
                const double self = *slot(p, cur, c);
                z[c] = fma(mk_, hop_sum(hd + 2 * col * HP_ST, off, cw), flip(self, g5));
                z[c] = fma(car, self, ib * z[c]);
                z[c] = fma(cai, slot(p, cur, c)[po], z[c]);
                z[c] = fma(cgr, *slot(p, prv, c), z[c]);
                z[c] = fma(cgi, slot(p, prv, c)[po], z[c]);
            }
            __syncwarp();  // the partner has read the previous vector, the warp its half spinors
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                *slot(p, prv, c) = z[c];
                if (ok && c < ncol) xn[((3 * sp + col0 + c) * V + site) * 2 + part] = z[c];
                const double zo = __shfl_xor_sync(0xffffffffu, z[c], 1);
                *slot(p, 2, c) = fma(cyi, zo, fma(cy.x, z[c], *slot(p, 2, c)));
            }
            __syncwarp();
        }
        if (i + 2 < kused) {
            grid_barrier_mono(a.bar, (unsigned)G * (++nbar), a.err, 1, LIM ? a.spin : LSPIN);
            if (*(volatile int*)a.err) return;
        }
    }
    for (int p = 0; p < a.npass; ++p) {
        const int site = SPW * (blockIdx.x + G * (wid + LW * p)) + sub;
        if (site >= a.V) continue;
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (c < ncol)
                reinterpret_cast<double*>(a.y)[((3 * sp + col0 + c) * V + site) * 2 + part] = *slot(p, 2, c);
    }
}

template <class A>
using CoopKernel = void (*)(A);

// the shared-memory opt-in of a kernel, once per device (attr_dev: the kernel's own record of devices)
template <class A>
void allow_smem(CoopKernel<A> kern, int rs, unsigned long long& attr_dev) {
    if (first_use_on_device(attr_dev))
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l2_smem(rs, L_MAXPASS));
}
unsigned long long l2_dev[2][2], regen_dev[2][2];  // k_l2_f64, k_regen_f64: RS = 1, 2; LIM

template <class A>
int launch_coop(CoopKernel<A> kern, A args, const Split& sp, unsigned long long& attr_dev, cudaStream_t st) {
    allow_smem(kern, sp.rs, attr_dev);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sp.G);
    cfg.blockDim = dim3(LT);
    cfg.dynamicSmemBytes = l2_smem(sp.rs, sp.npass);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, kern, args);
}

}  // namespace

bool l2_f64_ok(const Geom& g, int num_sms) {
    const Split sp = split_units(g.V, 2, num_sms);
    if (sp.npass > L_MAXPASS) return false;
    const CoopKernel<L2Args> kern = sp.rs == 1 ? k_l2_f64<1, false> : k_l2_f64<2, false>;
    allow_smem(kern, sp.rs, l2_dev[sp.rs - 1][0]);
    int dev = 0, coop = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, LT, l2_smem(sp.rs, sp.npass)) != cudaSuccess) {
        cudaGetLastError();  // (the per-step kernels report what is wrong, if anything)
        return false;
    }
    return split_fits(sp, num_sms, per_sm, coop != 0);
}

int launch_l2_f64(const double2* U64, const int* nbr, double2* const v[3], size_t vstep, double2* const w[3],
                  size_t wstep, KState* ks, double2* alpha, double2* beta, double2* gamma, double2* vscale, double mu,
                  double kappa, int k, double* partials, unsigned int* bar, const Geom& g, int num_sms,
                  cudaStream_t st, long long spin) {
    const Split sp = split_units(g.V, 2, num_sms);
    if (sp.npass > L_MAXPASS) return (int)cudaErrorInvalidValue;
    L2Args a;
    a.U = U64;
    a.nbr = nbr;
    for (int q = 0; q < 3; ++q) a.v[q] = v[q], a.w[q] = w[q];
    a.vstep = vstep, a.wstep = wstep;
    a.ks = ks;
    a.alpha = alpha, a.beta = beta, a.gamma = gamma, a.vscale = vscale;
    a.partA = partials;
    a.partC = partials + 4 * (size_t)sp.G;
    a.bar = bar;
    a.kappa = kappa, a.emu = exp(mu), a.emum = exp(-mu);
    a.V = g.V, a.k = k, a.npass = sp.npass;
    a.spin = spin;
    const bool lim = spin > 0;
    const CoopKernel<L2Args> kern = sp.rs == 1 ? (lim ? k_l2_f64<1, true> : k_l2_f64<1, false>)
                                               : (lim ? k_l2_f64<2, true> : k_l2_f64<2, false>);
    return launch_coop(kern, a, sp, l2_dev[sp.rs - 1][lim], st);
}

int launch_regen_f64(const double2* U64, const int* nbr, double2* const v[3], double2* y, const KState* ks,
                     const double2* coef, double mu, double kappa, unsigned int* bar, int* err, const Geom& g,
                     int num_sms, cudaStream_t st, long long spin) {
    const Split sp = split_units(g.V, 4, num_sms);
    if (sp.npass > L_MAXPASS) return (int)cudaErrorInvalidValue;
    R64Args a;
    a.U = U64;
    a.nbr = nbr;
    for (int q = 0; q < 3; ++q) a.v[q] = v[q];
    a.y = y;
    a.ks = ks;
    a.cf = coef;
    a.bar = bar;
    a.err = err;
    a.kappa = kappa, a.emu = exp(mu), a.emum = exp(-mu);
    a.V = g.V, a.npass = sp.npass;
    a.spin = spin;
    const bool lim = spin > 0;
    const CoopKernel<R64Args> kern = sp.rs == 1 ? (lim ? k_regen_f64<1, true> : k_regen_f64<1, false>)
                                                : (lim ? k_regen_f64<2, true> : k_regen_f64<2, false>);
    return launch_coop(kern, a, sp, regen_dev[sp.rs - 1][lim], st);
}

}  // namespace ovl
