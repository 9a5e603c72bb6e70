// Batched two-sided Lanczos solves: several right-hand sides on several gauge
// configurations (lattices of different sizes) in one sequence of launches,
// captured once as a CUDA graph.
//
// A sequence is one (configuration, right-hand side) pair.  Each batched kernel
// covers every sequence in one launch: its blocks are a concatenation of
// per-sequence block ranges (a device table maps a block to its sequence), so
// lattices of any size share the GPU in every step.  Reductions are per
// sequence: block partials and a ticket counter of their own, the last block
// of a sequence sums its partials in a fixed order and sets the coefficients
// (Sec. 4, Eq. 4.2).  A finished sequence (lucky breakdown, k reached) skips
// the rest of its work uniformly.  The links of a configuration are read by all
// of its right-hand sides in the same step and stay in L2 between them.
//
// Mixed precision (OVL_MIXED): pass 1 in FP32 with 12-real links (in-block sums
// of exact FP32 products in compensated pairs), pass 2 regenerates the basis
// from the pass-1 coefficients and accumulates y (Sec. 5) in double-float
// arithmetic (df32.cuh; native FP64 with OVL_PASS2_F64).  Otherwise
// FP64 throughout: one pass with the basis stored and the combination
// y = sum_i c_i v_i at the end, or, with OVL_TWO_PASS or when the basis would
// exceed 32 GiB, an FP64 pass 1 followed by the FP64 regeneration pass.
#include <algorithm>
#include <array>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "ctx.h"
#include "stencil_impl.cuh"

namespace ovl {

// Two-sided Lanczos passes near a breakdown for about one source in a hundred, and the result at a given k
// then hangs on pass 1's roundings: between two orders of the FP32 products such a source's results differ by
// 1e-9 to 1e-4 where all others agree to 1e-13.  A batch holds many sources, so its FP32 pass keeps the rounding
// that it always had (chained multiply-adds would take 2 % off a batch of 48).
template <class R> constexpr bool B_PF = sizeof(R) == 4;  // mul_link_pf

// per-step coefficients of the double-float regeneration (see k_b_regen_coef)
struct RegenCoefDf {
    float4 kb;        // kappa / beta_i (real; .x hi, .y lo)
    float4 cu, cl;    // cr of the upper and the lower spins {re hi, re lo, im hi, im lo}
    float4 cg, cc;    // cg; c_{i+1}
};

struct BSeq {
    Geom g;
    size_t n;                 // 12 V
    const void* U;            // pass-1 links: FP32-12 (float4) or FP64 (double2)
    const double2* U64;       // FP64 links (regeneration)
    const void* Udf;          // double-float links (regeneration of mixed solves)
    const int* nbr;           // [8][V] neighbour table of the lattice (regeneration)
    void* v[3];               // pass-1 ring (FP32 float4 pairs or FP64); unused with a stored basis
    void* w[3];
    void* t;
    void* s;
    double2* V;               // FP64 one-pass: stored basis, k + 1 vectors (else null)
    double2* r[3];            // FP64 regeneration ring (two-pass)
    double2* y;
    const double2* bR;        // b_perp^R (start of the regeneration)
    RegenCoefDf* rc;          // per-step coefficients of the double-float regeneration (mixed)
    KState* ks;
    double2* alpha;
    double2* beta;
    double2* gamma;
    double2* cvec;
    double2* vscale;
    double2* cf;              // recurrence coefficients of the step: alpha sv, conj(alpha) sw, gamma_{i-1} svp,
                              // conj(beta_{i-1}) swp
    double2* part;            // [nblk][4] block partials of the batched kernels
    unsigned int* cnt;        // ticket of this sequence
    int blk0[3], nblk[3];     // block range in the pass-1 launches, per site-block shape (64, 128, 256 sites)
    int tile0, ntile;         // tile range in the tiled launches (tiles of TT sites)
};

namespace {

// pass-1 site-block shapes (sites = threads per block), picked per batch by the autotuner
constexpr int NSHAPE = 3;
constexpr int SHAPE_SITES[NSHAPE] = {64, 128, 256};
constexpr int TT = 32;   // sites per tile of the direction-split kernels (one warp per direction)

template <class R> struct BVec;
template <> struct BVec<float> { using T = float4; };
template <> struct BVec<double> { using T = double2; };

template <class R> struct AccOf;
template <> struct AccOf<float> { using T = AccF; };
template <> struct AccOf<double> { using T = AccD; };

// accf_add(AccF, AccF), the pair addition of the block and sequence sums, is in df32.cuh
__device__ __forceinline__ AccF acc_shfl(AccF a, int o) {
    AccF r;
    r.hi = __shfl_xor_sync(0xffffffffu, a.hi, o);
    r.lo = __shfl_xor_sync(0xffffffffu, a.lo, o);
    return r;
}
__device__ __forceinline__ AccD accf_add(AccD a, AccD b) {
    AccD r;
    r.v = a.v + b.v;
    return r;
}
__device__ __forceinline__ AccD acc_shfl(AccD a, int o) {
    AccD r;
    r.v = __shfl_xor_sync(0xffffffffu, a.v, o);
    return r;
}
__device__ __forceinline__ double2 acc_store(AccF a) { return make_double2((double)a.hi, (double)a.lo); }
__device__ __forceinline__ double2 acc_store(AccD a) { return make_double2(a.v, 0.0); }
__device__ __forceinline__ AccF acc_load(double2 v, AccF) {
    AccF r;
    r.hi = (float)v.x;
    r.lo = (float)v.y;
    return r;
}
__device__ __forceinline__ AccD acc_load(double2 v, AccD) {
    AccD r;
    r.v = v.x;
    return r;
}

// Per-sequence reduction of NQ accumulators (in their own arithmetic: compensated FP32 pairs for FP32
// data, FP64 otherwise): warp trees, the block's warps in a fixed order into part[local], then the
// last block of the sequence (ticket) adds the partials of its nblk blocks in a fixed order.
// Returns true in the last block; out[] (FP64) is valid in every lane of warp 0 there.
template <int NQ, int NW, class A>
__device__ bool seq_reduce(A (&v)[NQ], double2* part, unsigned int* cnt, int local, int nblk, double (&out)[NQ]) {
    __shared__ double2 red[NQ][NW];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        A x = v[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x = accf_add(x, acc_shfl(x, o));
        if (lane == 0) red[q][wid] = acc_store(x);
    }
    __syncthreads();
    if (threadIdx.x < NQ) {
        const int q = threadIdx.x;
        A sacc = acc_load(red[q][0], A());
        for (int w = 1; w < NW; ++w) sacc = accf_add(sacc, acc_load(red[q][w], A()));
        part[(size_t)local * 4 + q] = acc_store(sacc);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned int t = atomicAdd(cnt, 1u);
        last = (t == (unsigned)nblk - 1);
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    // one warp per value (a warp takes several when the block has fewer warps than values): lanes
    // over the blocks, then the warp tree (fixed order)
    for (int qv = wid; qv < NQ; qv += NW) {
        A acc = acc_load(make_double2(0.0, 0.0), A());
        for (int b = lane; b < nblk; b += 32) acc = accf_add(acc, acc_load(__ldcg(&part[(size_t)b * 4 + qv]), A()));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc = accf_add(acc, acc_shfl(acc, o));
        if (lane == 0) red[qv][0] = acc_store(acc);
    }
    __syncthreads();
    if (wid == 0) {
        const double2 r = red[lane < NQ ? lane : 0][0];
        const double s = r.x + r.y;
#pragma unroll
        for (int q = 0; q < NQ; ++q) out[q] = __shfl_sync(0xffffffffu, s, q);
        if (lane == 0) *cnt = 0u;
    }
    return true;
}

// ---- the scalars of a step, by one warp (every lane gets the sums).  An FP64 instruction takes 64 cycles of
// its warp however few lanes take part, a library division 430 and a square root 680, and these chains are
// the tail of every step: real and imaginary parts go to lanes side by side, and the norms, their
// reciprocals and the divisions come from one reciprocal square root.
__device__ __forceinline__ double flip_sign(double x) {
    return __hiloint2double(__double2hiint(x) ^ (int)0x80000000u, __double2loint(x));
}
// alpha = conj(sw) w~^dag t from (re, im) = w~^dag t (sv is real): even lanes return its real part, odd lanes
// its imaginary part; r: lanes 0, 1 conj(alpha) sw, lanes 2, 3 alpha sv
__device__ __forceinline__ double alpha_scalars(double re, double im, double svr, double swr, double swi, double& r) {
    const int lane = threadIdx.x & 31;
    const bool q = lane & 1, first = lane < 2;
    const double al = fma(swr, q ? im : re, swi * (q ? flip_sign(re) : im));
    const double ao = __shfl_xor_sync(0xffffffffu, al, 1);
    const double ar = q ? ao : al, ai = q ? al : ao;
    const double m1 = first ? (q ? swi : swr) : svr, m2 = first ? (q ? flip_sign(swr) : swi) : 0.0;
    r = fma(first ? ar : al, m1, ai * m2);
    return al;
}
// beta = |v^|, gamma = delta / beta, sv' = 1 / beta, sw' = 1 / conj(gamma) = delta beta / |delta|^2 from
// delta = (re, im) and nv2 = |v^|^2: nv, rnv in every lane, g: lanes 0, 1 gamma, lanes 2, 3 sw';
// cn: lanes 0, 1 gamma sv, lanes 2, 3 beta sw (the next step's coefficients of the previous vectors)
__device__ __forceinline__ void beta_scalars(double re, double im, double nv2, double svr, double swr, double swi,
                                             double& nv, double& rnv, double& g, double& cn) {
    const int lane = threadIdx.x & 31;
    const bool q = lane & 1;
    const double nd2 = fma(im, im, re * re);
    const double r = rsqrt(q ? nd2 : nv2);  // even lanes 1 / |v^|, odd lanes 1 / |delta|
    const double r2 = r * (q ? r : nv2);    // |v^|, 1 / |delta|^2
    rnv = __shfl_sync(0xffffffffu, r, 0);
    nv = __shfl_sync(0xffffffffu, r2, 0);
    const double f = nv * __shfl_sync(0xffffffffu, r2, 1);
    g = (q ? im : re) * (lane < 2 ? rnv : f);
    cn = (lane < 2 ? g : nv) * (lane < 2 ? svr : (q ? swi : swr));
}
// lucky (1) or serious (2) breakdown from the squared norms; an2: largest |A v_i|^2 so far
__device__ __forceinline__ int breakdown(double re, double im, double nv2, double nw2, double an2) {
    if (nv2 <= 1e-26 * fmax(an2, 1e-300)) return 1;  // |v^| <= 1e-13 max |A v_i|
    return fma(im, im, re * re) <= 1e-28 * nv2 * nw2 ? 2 : 0;  // |w^^dag v^| <= 1e-14 |v^| |w^|
}

// Programmatic dependent launch: the batched kernels of one solve follow each other on one
// stream and are launched with programmatic stream serialisation, so a kernel's blocks may be
// scheduled while the previous kernel drains.  Each kernel waits here (full completion and memory
// visibility of the previous grid) before it reads anything the previous kernel wrote, and lets
// the next kernel be scheduled once all of its own blocks have started.
__device__ __forceinline__ void pdl_wait_and_release() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class R>
__device__ __forceinline__ void* vslot(const BSeq& q, int j, bool wvec) {
    if (!wvec && q.V) return q.V + (size_t)j * q.n;
    return wvec ? q.w[j % 3] : q.v[j % 3];
}

// t = sv A v~_i, s = sw A^dag w~_i at every site of every running sequence; alpha_i = w_i^dag t.
// The grid's y index splits the two stencils (y = 0: t and the alpha partials; y = 1: s), so a
// thread carries one accumulator spinor instead of two (fewer registers: more warps per SM).
// Both run the same copy of the stencil (two copies cost instruction fetches: batch of 48 252.6 -> 250.7 ms).
// The last step's s (i = klast) is not used, so the y = 1 blocks may skip it once the sequence
// is marked done.
// The FP32 form is compiled for 768 resident threads per SM (at most 80 registers): measured on the
// 48-sequence batch, pass 1 137.1 -> 134.3 ms (64-site blocks) and 145.4 -> 134.7 ms (128).
template <int LF, class R, int SH>
__global__ void __launch_bounds__(SHAPE_SITES[SH], LF == LINK_F64 ? 1 : 768 / SHAPE_SITES[SH]) k_b_pair(
    const BSeq* __restrict__ S, const int* __restrict__ bseq, int i, int klast, HopCoef<R> hv, HopCoef<R> hw) {
    using VT = typename BVec<R>::T;
    const BSeq& q = S[bseq[blockIdx.x]];  // set-up data, not written by the solve
    KState* ks = q.ks;
    pdl_wait_and_release();
    if (ks->done || ks->status) return;
    constexpr int BT = SHAPE_SITES[SH];
    const int local = blockIdx.x - q.blk0[SH];
    const int site = local * BT + threadIdx.x;
    const VT* vi = (const VT*)vslot<R>(q, i, false);
    const VT* wi = (const VT*)vslot<R>(q, i, true);
    const bool second = blockIdx.y == 1;  // s = sw A^dag w~
    typename AccOf<R>::T a[3];
    if (site < q.g.V) {
        const VT* const xs[1] = {second ? wi : vi};
        HopCoef<R> hcs[1] = {hv};
        hcs[0].f[3] = second ? hw.f[3] : hv.f[3];
        hcs[0].b[3] = second ? hw.b[3] : hv.b[3];
        const double2 scale = second ? ks->sw : ks->sv;
        const cx<R> cs = mk((R)scale.x, (R)scale.y);
        Spinor<R> acc[1], self;
        apply_site<LF, R, 1, false, B_PF<R>>(q.g, site, q.U, xs, acc, hcs);
        load_spinor(xs[0], q.g.V, site, self);
        finish_site(acc[0], self, true);
#pragma unroll
        for (int sp = 0; sp < 4; ++sp)
#pragma unroll
            for (int c = 0; c < 3; ++c) acc[0].s[sp][c] = cs * acc[0].s[sp][c];
        store_spinor((VT*)(second ? q.s : q.t), q.g.V, site, acc[0]);
        if (!second) {
            load_spinor(wi, q.g.V, site, self);  // w~ at the own site: alpha = conj(sw) w~^dag t
#pragma unroll
            for (int sp = 0; sp < 4; ++sp)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    acc_cdot(a, self.s[sp][c], acc[0].s[sp][c]);
                    acc_norm2(a[2], acc[0].s[sp][c]);
                }
        }
    }
    if (second) return;
    double o[3];
    if (seq_reduce<3, BT / 32>(a, q.part, q.cnt, local, q.nblk[SH], o) && threadIdx.x < 32) {
        const int lane = threadIdx.x;
        double r;
        const double al = alpha_scalars(o[0], o[1], ks->sv.x, ks->sw.x, ks->sw.y, r);
        if (lane < 4) reinterpret_cast<double*>(q.cf + (lane < 2 ? 1 : 0))[lane & 1] = r;
        if (lane < 2) reinterpret_cast<double*>(q.alpha + i)[lane] = al;
        if (lane == 0) {
            ks->red[0].x = fmax(ks->red[0].x, o[2]);  // max |A v_i|^2
            ks->kused = i + 1;
            if (i >= klast) ks->done = 1;
        }
    }
}

// 16-byte chunks of a device-layout vector: FP32 float4 = two complex, FP64 double2 = one
template <class R> struct Chunk;
template <> struct Chunk<float> {
    static constexpr int N = 6, P = 2;
    static __device__ __forceinline__ void split(const float4 v, cx<float> (&z)[2]) {
        z[0] = mk(v.x, v.y);
        z[1] = mk(v.z, v.w);
    }
    static __device__ __forceinline__ float4 join(const cx<float> (&z)[2]) {
        return make_float4(z[0].r, z[0].i, z[1].r, z[1].i);
    }
};
template <> struct Chunk<double> {
    static constexpr int N = 12, P = 1;
    static __device__ __forceinline__ void split(const double2 v, cx<double> (&z)[1]) { z[0] = mk(v.x, v.y); }
    static __device__ __forceinline__ double2 join(const cx<double> (&z)[1]) { return make_double2(z[0].r, z[0].i); }
};

// v^ = t - alpha v_i - gamma_{i-1} v_{i-1}, w^ = s - conj(alpha) w_i - conj(beta_{i-1}) w_{i-1};
// w^^dag v^, |v^|^2, |w^|^2 -> beta_i, gamma_i, the scales, breakdown checks (Eq. 4.2).  Element by
// element: one 16-byte chunk of each operand at a time (few registers, many warps per SM).
// The FP32 form is compiled for 1536 resident threads per SM (at most 40 registers): measured on the
// 48-sequence batch, pass 1 134.9 -> 130.9 ms (128-site blocks).
template <class R, int SH>
__global__ void __launch_bounds__(SHAPE_SITES[SH], sizeof(R) == 4 ? 1536 / SHAPE_SITES[SH] : 1)
    k_b_lstep(const BSeq* __restrict__ S, const int* __restrict__ bseq, int i) {
    using VT = typename BVec<R>::T;
    using CH = Chunk<R>;
    constexpr int P = CH::P;
    const BSeq& q = S[bseq[blockIdx.x]];  // set-up data, not written by the solve
    KState* ks = q.ks;
    pdl_wait_and_release();
    if (ks->done || ks->status) return;
    __shared__ cx<R> cf[4];
    if (threadIdx.x < 4) {
        const double2 c = q.cf[threadIdx.x];
        cf[threadIdx.x] = mk((R)c.x, (R)c.y);
    }
    __syncthreads();
    constexpr int BT = SHAPE_SITES[SH];
    const int local = blockIdx.x - q.blk0[SH];
    const int site = local * BT + threadIdx.x;
    typename AccOf<R>::T a[4];
    if (site < q.g.V) {
        const size_t V = (size_t)q.g.V;
        const VT* tp = (const VT*)q.t;
        const VT* sp_ = (const VT*)q.s;
        const VT* vp = (const VT*)vslot<R>(q, i, false);
        const VT* wp = (const VT*)vslot<R>(q, i, true);
        const VT* vmp = (const VT*)vslot<R>(q, i > 0 ? i - 1 : i, false);
        const VT* wmp = (const VT*)vslot<R>(q, i > 0 ? i - 1 : i, true);
        VT* vn = (VT*)vslot<R>(q, i + 1, false);
        VT* wn = (VT*)vslot<R>(q, i + 1, true);
        const cx<R> c0 = cf[0], c1 = cf[1], c2 = cf[2], c3 = cf[3];
#pragma unroll 2
        for (int ch = 0; ch < CH::N; ++ch) {
            const size_t e = (size_t)ch * V + site;
            cx<R> t[P], s[P], vv[P], ww[P], vm[P], wm[P];
            CH::split(__ldg(tp + e), t);
            CH::split(__ldg(sp_ + e), s);
            CH::split(__ldg(vp + e), vv);
            CH::split(__ldg(wp + e), ww);
            if (i > 0) {
                CH::split(__ldg(vmp + e), vm);
                CH::split(__ldg(wmp + e), wm);
            }
#pragma unroll
            for (int p = 0; p < P; ++p) {
                cx<R> x = t[p] - c0 * vv[p];
                cx<R> y = s[p] - c1 * ww[p];
                if (i > 0) {
                    x = x - c2 * vm[p];
                    y = y - c3 * wm[p];
                }
                t[p] = x;
                s[p] = y;
                acc_cdot(a, y, x);
                acc_norm2(a[2], x);
                acc_norm2(a[3], y);
            }
            vn[e] = CH::join(t);
            wn[e] = CH::join(s);
        }
    }
    double o[4];
    if (seq_reduce<4, BT / 32>(a, q.part, q.cnt, local, q.nblk[SH], o) && threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const int bk = breakdown(o[0], o[1], o[2], o[3], ks->red[0].x);
        if (bk) {
            if (lane == 0) {
                ks->done = 1;
                if (bk == 2) ks->bdstep = i + 1;
            }
        } else {
            const double2 sv = ks->sv, sw = ks->sw;
            double nv, rnv, g, cn;
            beta_scalars(o[0], o[1], o[2], sv.x, sw.x, sw.y, nv, rnv, g, cn);
            __syncwarp();
            if (lane < 2) reinterpret_cast<double*>(q.gamma + i)[lane] = g;
            else if (lane < 4) reinterpret_cast<double*>(&ks->sw)[lane & 1] = g;
            if (lane < 4) reinterpret_cast<double*>(q.cf + 2)[lane] = cn;
            if (lane == 0) {
                q.beta[i] = make_double2(nv, 0.0);
                ks->svp = sv;
                ks->swp = sw;
                ks->sv = q.vscale[i + 1] = make_double2(rnv, 0.0);
            }
        }
    }
}

// ---- persistent batched pass 1 (all sites of the batch resident at once) ----------------------
// One cooperative launch runs the whole FP32 pass 1 of every sequence: one thread per site, blocks
// of BP1_T sites, each block within one sequence.  Per step: phase A, t = sv A v~_i and
// s = sw A^dag w~_i at the own site (kept in registers), block partials of w~^dag t and |t|^2;
// the sequence's blocks meet at a bounded barrier (a monotonic counter per sequence); every block
// sums the sequence's partials in the same fixed order, so all of them hold the same alpha_i;
// phase C, the recurrence of Eq. 4.2 at the own site (v^, w^ stored: the neighbours' next
// stencil reads them), partials of w^^dag v^, |v^|^2, |w^|^2; second barrier; every block forms
// beta_i, gamma_i, the scales and the breakdown decisions, identically.  Sequences finish
// independently.  Vector loads go through L2 (.cg): the ring slots are rewritten during the launch.
constexpr int BP1_T = 128;
constexpr long long BP1_SPIN = 20000000;  // polls before a barrier wait gives up (sets ks->timeout)

struct BP1Args {
    const BSeq* S;
    const int* bseq;      // block -> sequence (blocks of BP1_T sites: the pass-1 shape 1 tables)
    unsigned int* bar;    // one barrier counter per sequence, zero at launch
    int k;
    HopCoef<float> hv, hw;
};

// Block sum of NQ compensated pairs into part[local * 4 + q] (warp trees, then the warps in order).
template <int NQ>
__device__ __forceinline__ void bp1_block_partial(AccF (&v)[NQ], double2* part, int local) {
    __shared__ double2 red[NQ][BP1_T / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        AccF x = v[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x = accf_add(x, acc_shfl(x, o));
        if (lane == 0) red[q][wid] = acc_store(x);
    }
    __syncthreads();
    if (threadIdx.x < NQ) {
        const int q = threadIdx.x;
        AccF sacc = acc_load(red[q][0], AccF());
        for (int w = 1; w < BP1_T / 32; ++w) sacc = accf_add(sacc, acc_load(red[q][w], AccF()));
        part[(size_t)local * 4 + q] = acc_store(sacc);
    }
}

// The sequence's sums of NQ values over its nblk block partials, in a fixed order (lanes over the
// blocks, then the warp tree), one warp per value; out (shared) is valid in all threads on return.
template <int NQ>
__device__ __forceinline__ void bp1_seq_sum(const double2* part, int nblk, double* out) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int qv = wid; qv < NQ; qv += BP1_T / 32) {
        AccF acc = acc_load(make_double2(0.0, 0.0), AccF());
        for (int b = lane; b < nblk; b += 32) acc = accf_add(acc, acc_load(__ldcg(&part[(size_t)b * 4 + qv]), AccF()));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc = accf_add(acc, acc_shfl(acc, o));
        if (lane == 0) {
            const double2 r = acc_store(acc);
            out[qv] = r.x + r.y;
        }
    }
    __syncthreads();
}

__device__ __forceinline__ cx<float> f32c(cx<double> z) { return mk((float)z.r, (float)z.i); }

template <int LF>
__global__ void __launch_bounds__(BP1_T, 3) k_bp1(BP1Args a) {
    const int sidx = a.bseq[blockIdx.x];
    const BSeq& q = a.S[sidx];
    KState* ks = q.ks;
    if (ks->done || ks->status) return;  // the whole sequence leaves (written before this launch)
    __shared__ cx<float> cs[2];          // sv, sw of the current step
    __shared__ cx<float> cc[4];          // alpha sv, conj(alpha) sw, gamma_{i-1} svp, conj(beta_{i-1}) swp
    __shared__ double osum[4];
    __shared__ int sdone;
    const int local = blockIdx.x - q.blk0[1], nblk = q.nblk[1];
    const int site = local * BP1_T + threadIdx.x;
    const bool ok = site < q.g.V;
    const int V = q.g.V;
    unsigned int* bar = a.bar + sidx;
    int* err = &ks->timeout;
    double2* partA = q.part;
    double2* partC = q.part + (size_t)nblk * 4;
    // recurrence scalars in FP64 (identical in every block of the sequence; sv is real), in shared memory: no
    // registers between the uses
    __shared__ double sc[7];             // sv, sw (re, im), svp, swp (re, im); max |A v_i|^2
    __shared__ int steps[2];             // steps taken, step of a serious breakdown
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        sc[0] = ks->sv.x, sc[1] = ks->sw.x, sc[2] = ks->sw.y;
        sc[3] = ks->svp.x, sc[4] = ks->swp.x, sc[5] = ks->swp.y;
        sc[6] = ks->anorm * ks->anorm;
        steps[0] = 0, steps[1] = -1;
        cs[0] = mk((float)sc[0], 0.f);
        cs[1] = mk((float)sc[1], (float)sc[2]);
        cc[2] = cc[3] = mk(0.f, 0.f);
    }
    __syncthreads();
    unsigned int nb = 0;
    for (int i = 0; i < a.k; ++i) {
        const float4* vi = (const float4*)q.v[i % 3];
        const float4* wi = (const float4*)q.w[i % 3];
        // ---- phase A
        AccF pa[3];
        Spinor<float> t, s;
        if (ok) {
            const float4* const xs[2] = {vi, wi};
            const HopCoef<float> hcs[2] = {a.hv, a.hw};
            Spinor<float> acc[2], self[2];
            apply_site<LF, float, 2, true, B_PF<float>>(q.g, site, q.U, xs, acc, hcs);
            load_spinor_cg(vi, V, site, self[0]);
            load_spinor_cg(wi, V, site, self[1]);
            finish_site(acc[0], self[0], true);
            finish_site(acc[1], self[1], true);
            t = acc[0];
            s = acc[1];
            const cx<float> fsv = cs[0], fsw = cs[1];
#pragma unroll
            for (int sp = 0; sp < 4; ++sp)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    t.s[sp][c] = fsv * t.s[sp][c];
                    s.s[sp][c] = fsw * s.s[sp][c];
                    acc_cdot(pa, self[1].s[sp][c], t.s[sp][c]);
                    acc_norm2(pa[2], t.s[sp][c]);
                }
        }
        bp1_block_partial<3>(pa, partA, local);
        grid_barrier_mono(bar, (unsigned)nblk * (++nb), err, 1, BP1_SPIN);
        if (*(volatile int*)err) return;
        bp1_seq_sum<3>(partA, nblk, osum);
        if (wid == 0) {
            double r;
            const double al = alpha_scalars(osum[0], osum[1], sc[0], sc[1], sc[2], r);
            if (lane < 4) reinterpret_cast<float*>(cc + (lane < 2 ? 1 : 0))[lane & 1] = (float)r;
            if (local == 0 && lane < 2) reinterpret_cast<double*>(q.alpha + i)[lane] = al;
        } else if (threadIdx.x == 32) {
            sc[6] = fmax(sc[6], osum[2]);
            steps[0] = i + 1;
        }
        if (i == a.k - 1) break;
        __syncthreads();
        // ---- phase C: v^ = t - alpha v_i - gamma_{i-1} v_{i-1}, w^ likewise (Eq. 4.2)
        AccF pc[4];
        if (ok) {
            const cx<float> ca = cc[0], da = cc[1], cg = cc[2], db = cc[3];
            Spinor<float> vv, ww, vm, wm;
            load_spinor_cg(vi, V, site, vv);
            load_spinor_cg(wi, V, site, ww);
            if (i > 0) {
                load_spinor_cg((const float4*)q.v[(i + 2) % 3], V, site, vm);
                load_spinor_cg((const float4*)q.w[(i + 2) % 3], V, site, wm);
            }
#pragma unroll
            for (int sp = 0; sp < 4; ++sp)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    cx<float> x = t.s[sp][c] - ca * vv.s[sp][c];
                    cx<float> y = s.s[sp][c] - da * ww.s[sp][c];
                    if (i > 0) {
                        x = x - cg * vm.s[sp][c];
                        y = y - db * wm.s[sp][c];
                    }
                    t.s[sp][c] = x;
                    s.s[sp][c] = y;
                    acc_cdot(pc, y, x);
                    acc_norm2(pc[2], x);
                    acc_norm2(pc[3], y);
                }
            store_spinor((float4*)q.v[(i + 1) % 3], V, site, t);
            store_spinor((float4*)q.w[(i + 1) % 3], V, site, s);
        }
        bp1_block_partial<4>(pc, partC, local);
        grid_barrier_mono(bar, (unsigned)nblk * (++nb), err, 1, BP1_SPIN);
        if (*(volatile int*)err) return;
        bp1_seq_sum<4>(partC, nblk, osum);
        double nv = 0.0, rnv = 0.0, g = 0.0, cn = 0.0;
        if (wid == 0) {
            beta_scalars(osum[0], osum[1], osum[2], sc[0], sc[1], sc[2], nv, rnv, g, cn);
        } else if (wid == 1) {
            const int bk = breakdown(osum[0], osum[1], osum[2], osum[3], sc[6]);
            if (lane == 0) {
                sdone = bk;
                if (bk == 2) steps[1] = i + 1;
            }
        }
        __syncthreads();
        if (sdone) break;
        if (wid == 0) {
            const double swr = __shfl_sync(0xffffffffu, g, 2), swi = __shfl_sync(0xffffffffu, g, 3);
            if (lane < 4) reinterpret_cast<float*>(cc + 2)[lane] = (float)cn;
            if (lane == 0) {
                sc[3] = sc[0], sc[4] = sc[1], sc[5] = sc[2];
                sc[0] = rnv, sc[1] = swr, sc[2] = swi;
                cs[0] = mk((float)rnv, 0.f);
                cs[1] = mk((float)swr, (float)swi);
            }
            if (local == 0) {
                if (lane < 2) reinterpret_cast<double*>(q.gamma + i)[lane] = g;
                if (lane == 0) {
                    q.beta[i] = make_double2(nv, 0.0);
                    q.vscale[i + 1] = make_double2(rnv, 0.0);
                }
            }
        }
        __syncthreads();
    }
    if (local == 0 && threadIdx.x == 32) {
        ks->sv = make_double2(sc[0], 0.0);
        ks->sw = make_double2(sc[1], sc[2]);
        ks->svp = make_double2(sc[3], 0.0);
        ks->swp = make_double2(sc[4], sc[5]);
        ks->kused = steps[0];
        ks->done = 1;
        ks->anorm = sqrt(sc[6]);
        if (steps[1] >= 0) ks->bdstep = steps[1];
    }
}

// Regeneration (Sec. 5): r_{i+1} = ((A - alpha_i) r_i - gamma_{i-1} r_{i-1}) / beta_i, y += c_{i+1} r_{i+1}:
// in double-float (k_b_regen_df, mixed solves) or in FP64 (k_b_regen, k_b_regen2).

// ---- double-float regeneration ----------------------------------------------------------------
// Vectors (r, y) of the pass are stored with the two spins of a half spinor side by side: chunk
// (P * 3 + colour) * 2 + part of a site is the float4 {hi of spin 2P, hi of spin 2P + 1, lo, lo} of the
// real (part 0) or imaginary (part 1) part, the operand layout of the packed FP32x2 arithmetic.
//
// Coefficients of a step, formed once per sequence (k_b_regen_coef) and stored as double-float: with
// S the sum of the hops (e^{+-mu} on the temporal ones, kappa taken out), A r = r - kappa S on the upper
// spins and -(r - kappa S) on the lower, so
//   r_{i+1} = cr r_i -+ (kappa / beta_i) S + cg r_{i-1},  cr = (+-1 - alpha_i) / beta_i, cg = -gamma_{i-1} / beta_i.

__device__ __forceinline__ float4 df4(cx<double> z) {
    const df r(z.r), i(z.i);
    return make_float4(r.hi, r.lo, i.hi, i.lo);
}

// grid (steps / 128, sequences)
__global__ void k_b_regen_coef(const BSeq* __restrict__ S, double kappa) {
    const BSeq& q = S[blockIdx.y];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (q.ks->status || i + 1 >= q.ks->kused) return;
    const double ib = 1.0 / q.beta[i].x;  // beta_i is real
    const cx<double> a = ib * d2c(q.alpha[i]);
    RegenCoefDf c;
    c.kb = df4(mk(ib * kappa, 0.0));
    c.cu = df4(mk(ib - a.r, -a.i));
    c.cl = df4(mk(-ib - a.r, -a.i));
    c.cg = i > 0 ? df4(-(ib * d2c(q.gamma[i - 1]))) : make_float4(0.f, 0.f, 0.f, 0.f);
    c.cc = df4(d2c(q.cvec[i + 1]));
    q.rc[i] = c;
}

// r_1 = b_perp / |b_perp|, y += c_1 r_1 in FP64, both then split into the packed layout (y in place: a
// thread owns its site); one launch for all sequences, blocks as in the pass-1 shape of 128 sites.
__global__ void __launch_bounds__(128) k_b_regen_start(const BSeq* __restrict__ S, const int* __restrict__ bseq) {
    const BSeq& q = S[bseq[blockIdx.x]];
    const int site = (blockIdx.x - q.blk0[1]) * 128 + threadIdx.x;
    if (site >= q.g.V) return;
    const size_t V = (size_t)q.g.V;
    const bool run = !q.ks->status && q.ks->nR != 0.0;
    const cx<double> sv = mk(run ? 1.0 / q.ks->nR : 0.0, 0.0), c0 = d2c(q.cvec[0]);
    df yr[12], yi[12];
    float4* r0 = reinterpret_cast<float4*>(q.r[0]);
    float4* yo = reinterpret_cast<float4*>(q.y);
#pragma unroll
    for (int P = 0; P < 2; ++P)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            cx<df> z[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = 3 * (2 * P + h) + a;
                cx<double> y = d2c(q.y[(size_t)c * V + site]);
                if (run) {
                    const cx<double> v = sv * d2c(q.bR[(size_t)c * V + site]);
                    cfma(y, c0, v);
                    z[h] = mk(df(v.r), df(v.i));
                }
                yr[c] = df(y.r);
                yi[c] = df(y.i);
            }
            if (run) {
                const size_t e = (size_t)(P * 3 + a) * 2 * V + site;
                r0[e] = make_float4(z[0].r.hi, z[1].r.hi, z[0].r.lo, z[1].r.lo);
                r0[e + V] = make_float4(z[0].i.hi, z[1].i.hi, z[0].i.lo, z[1].i.lo);
            }
        }
#pragma unroll
    for (int P = 0; P < 2; ++P)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int c0_ = 6 * P + a, c1_ = 6 * P + 3 + a;
            const size_t e = (size_t)(P * 3 + a) * 2 * V + site;
            yo[e] = make_float4(yr[c0_].hi, yr[c1_].hi, yr[c0_].lo, yr[c1_].lo);
            yo[e + V] = make_float4(yi[c0_].hi, yi[c1_].hi, yi[c0_].lo, yi[c1_].lo);
        }
}

// y back to FP64 in the component layout (in place)
__global__ void __launch_bounds__(128) k_b_regen_out(const BSeq* __restrict__ S, const int* __restrict__ bseq) {
    const BSeq& q = S[bseq[blockIdx.x]];
    const int site = (blockIdx.x - q.blk0[1]) * 128 + threadIdx.x;
    if (site >= q.g.V) return;
    const size_t V = (size_t)q.g.V;
    float4 v[12];
    const float4* yi = reinterpret_cast<const float4*>(q.y);
#pragma unroll
    for (int c = 0; c < 12; ++c) v[c] = yi[(size_t)c * V + site];
#pragma unroll
    for (int P = 0; P < 2; ++P)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float4 re = v[(P * 3 + a) * 2], im = v[(P * 3 + a) * 2 + 1];
            q.y[(size_t)(6 * P + a) * V + site] =
                make_double2((double)re.x + (double)re.z, (double)im.x + (double)im.z);
            q.y[(size_t)(6 * P + 3 + a) * V + site] =
                make_double2((double)re.y + (double)re.w, (double)im.y + (double)im.w);
        }
}

// real and imaginary sums of a pair of spins
struct CAcc2 {
    dfacc2 r, i;
};

// 16-byte asynchronous copy global -> shared (completion: cp.async.wait_group, a hardware wait)
__device__ __forceinline__ void cp_async16(float4* dst, const float4* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Projected half spinor h (both spins packed): (1 + S gamma_NU) psi, spins 0 and 1, of the spinor in the
// slots p[0], p[T], ... p[11 T]; sg the signs of the lower components in them (+-1, from the sense).
template <int NU, int T>
__device__ __forceinline__ void project_dfx(const float4* p, float2 sg, CAcc2 (&h)[3]) {
    constexpr bool HI2 = NU >= 2, IM = (NU & 1) == 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float4 ur = p[2 * a * T], ui = p[(2 * a + 1) * T];
        float4 lr = p[(6 + 2 * a) * T], li = p[(7 + 2 * a) * T];
        if (!HI2) {  // spin 0 takes the lower spin 3, spin 1 the lower spin 2
            lr = make_float4(lr.y, lr.x, lr.w, lr.z);
            li = make_float4(li.y, li.x, li.w, li.z);
        }
        h[a].r.s = make_float2(ur.x, ur.y), h[a].r.e = make_float2(ur.z, ur.w);
        h[a].i.s = make_float2(ui.x, ui.y), h[a].i.e = make_float2(ui.z, ui.w);
        const float2 lrh = make_float2(lr.x, lr.y), lrl = make_float2(lr.z, lr.w);
        const float2 lih = make_float2(li.x, li.y), lil = make_float2(li.z, li.w);
        if (IM) {  // + sg i (lower)
            dfacc2_add_signed(h[a].r, f2_neg(sg), lih, lil);
            dfacc2_add_signed(h[a].i, sg, lrh, lrl);
        } else {
            dfacc2_add_signed(h[a].r, sg, lrh, lrl);
            dfacc2_add_signed(h[a].i, sg, lih, lil);
        }
    }
}

// One thread per site and sequence: the eight hops one after the other, the four spins' sums in
// registers (double-float, spins packed in pairs), then the recurrence and y in the same thread.
// The hop loop is rolled (direction and sense are uniform), the link product is one piece of code for U
// and U^dag (row or column addressing and the sign of the imaginary parts), one link row at a time.
// Bound by the FP32 pipe: 10800 FP32 operations per site and step (per hop 12 projection sums of 8, 12
// sums of 6 products at 64, 24 spin sums of 8; per part of an output component 52 for the recurrence, 30
// for y and three renormalisations of 3; the temporal coefficients 168).  With the loads left to the hop
// that uses them a warp stood on them 70 % of its time at 16 warps per SM (415 us below); each thread's
// copies for the next hop now go to its own slots of shared memory while it computes the present one (no
// block barrier anywhere).
// Measured on the 48-sequence batch (706752 sites): 290 us per launch, 26.3 Top/s = 0.65 of the FP32 issue
// rate, FMA pipe 67 % busy; the form before this one (eight hop warps per 32-site tile, half spinors
// through shared memory, scalar instructions) took 552.  16^3 x 32, one source: 121 -> 64 us;
// 12 sources on 8^4: 59.8 -> 28.9 us.  Against the FP64 pass after 480 steps: 1.7 ... 2.0e-14 (2.0 ...
// 2.3e-14 before; y's low part is what that error is made of).  Blocks of 64: 32 and 128 differ by less
// than 1 %; four sequences of a lattice in one block were no faster (their links meet in L2 either way).
constexpr int RD_T = 64;  // sites per block
constexpr size_t RD_SM = 21 * RD_T * sizeof(float4);
template <int MINB>
__global__ void __launch_bounds__(RD_T, 2 * MINB) k_b_regen_df(const BSeq* __restrict__ S,
                                                               const int2* __restrict__ work, int i, df emu,
                                                               df emum) {
    const int2 wk = work[blockIdx.x];  // sequence, first site (set-up data)
    const BSeq& q = S[wk.x];
    const size_t V = (size_t)q.g.V;
    // (threads past the lattice take its last site and write nothing)
    const bool own = wk.y + (int)threadIdx.x < q.g.V;
    const int site = own ? wk.y + (int)threadIdx.x : q.g.V - 1;
    int ne = __ldg(q.nbr + site), nx = __ldg(q.nbr + 4 * V + site);
    pdl_wait_and_release();
    const float4* __restrict__ x = reinterpret_cast<const float4*>(q.r[i % 3]);
    const float4* __restrict__ U = reinterpret_cast<const float4*>(q.Udf);
    // this thread's operands of a hop: 12 chunks of the neighbour's spinor, then 9 link elements
    extern __shared__ __align__(16) float4 rd_sm[];
    float4* ps = rd_sm + threadIdx.x;
    float4* us = ps + 12 * RD_T;
    // copies of hop hh's spinor / link row a (hop order: direction hh >> 1, forward first)
    auto fetch_spinor = [&](int ne) {
        const float4* xb = x + (ne < 0 ? ~ne : ne);
#pragma unroll
        for (int c = 0; c < 12; ++c) cp_async16(ps + c * RD_T, xb + (size_t)c * V);
    };
    auto fetch_row = [&](int hh, int ne, int a) {
        const bool fwd = (hh & 1) == 0;
        const float4* u = U + (size_t)(hh >> 1) * 9 * V + (fwd ? site : (ne < 0 ? ~ne : ne));
        const size_t srow = fwd ? 3 * V : V, scol = fwd ? V : 3 * V;  // U: row a; U^dag: column a
#pragma unroll
        for (int k = 0; k < 3; ++k) cp_async16(us + (3 * a + k) * RD_T, u + (size_t)a * srow + (size_t)k * scol);
    };
    const float2 one = make_float2(1.f, 1.f);
    CAcc2 up[3], lw[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        up[a].r.s = up[a].r.e = up[a].i.s = up[a].i.e = make_float2(0.f, 0.f);
        lw[a] = up[a];
    }
    // the first hop's copies leave before the state is read (a finished sequence only drops them)
    fetch_spinor(ne);
    cp_async_commit();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        fetch_row(0, ne, a);
        cp_async_commit();
    }
    if (q.ks->status || i + 1 >= q.ks->kused) {
        cp_async_wait<0>();
        return;
    }
    const float4* __restrict__ xm = reinterpret_cast<const float4*>(q.r[(i + 2) % 3]);
#pragma unroll 1
    for (int hh = 0; hh < 8; ++hh) {
        const int nu = hh >> 1;
        const bool fwd = (hh & 1) == 0;
        if (hh == 4) {  // the lower sums were kept as spins (3, 2) for nu < 2; (2, 3) from here
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                lw[a].r.s = make_float2(lw[a].r.s.y, lw[a].r.s.x);
                lw[a].r.e = make_float2(lw[a].r.e.y, lw[a].r.e.x);
                lw[a].i.s = make_float2(lw[a].i.s.y, lw[a].i.s.x);
                lw[a].i.e = make_float2(lw[a].i.e.y, lw[a].i.e.x);
            }
        }
        const bool flip = ne < 0;  // the hop crosses the antiperiodic boundary
        ne = nx;
        if (hh < 6) nx = __ldg(q.nbr + (size_t)(((hh + 2) >> 1) + (fwd ? 0 : 4)) * V + site);
        const float fs = fwd ? 1.f : -1.f;
        // signs of the projected lower components in spins 0, 1 (chiral basis)
        const float2 sg = make_float2(nu == 3 ? fs : -fs, nu == 0 ? -fs : fs);
        CAcc2 h[3];
        // groups in flight: this hop's spinor and three link rows, one group each; every group is
        // replaced by the next hop's once it is consumed, so three younger ones are always behind
        cp_async_wait<3>();
        switch (nu) {
            case 0: project_dfx<0, RD_T>(ps, sg, h); break;
            case 1: project_dfx<1, RD_T>(ps, sg, h); break;
            case 2: project_dfx<2, RD_T>(ps, sg, h); break;
            default: project_dfx<3, RD_T>(ps, sg, h); break;
        }
        // behind the last hop come the recurrence's operands: the own r_i in the spinor's slots, the first
        // nine chunks of r_{i-1} in the link's
        fetch_spinor(hh < 7 ? ne : site);
        cp_async_commit();
        // signs of the half spinor in the lower spins: (from spin 0, from spin 1)
        const float sA = fs, sB = (nu == 0 || nu == 3) ? fs : -fs;
        const float2 lsg = nu < 2 ? make_float2(sB, sA) : make_float2(sA, sB);
        const bool im = (nu & 1) == 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            CAcc2 o;
            cp_async_wait<3>();
            const float4 u3[3] = {us[3 * a * RD_T], us[(3 * a + 1) * RD_T], us[(3 * a + 2) * RD_T]};
            if (hh < 7) {
                fetch_row(hh + 1, ne, a);
            } else if (i > 0) {
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    cp_async16(us + (3 * a + k) * RD_T, xm + (size_t)(3 * a + k) * V + site);
            }
            cp_async_commit();
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float4 v = u3[k];
                const float2 rh = f2_dup(v.x), rl = f2_dup(v.y);
                const float2 ih = f2_dup(fs * v.z), il = f2_dup(fs * v.w);  // U^dag: conjugate
                if (k == 0) {
                    dfacc2_first(o.r, rh, rl, h[k].r.s, h[k].r.e);
                    dfacc2_first(o.i, rh, rl, h[k].i.s, h[k].i.e);
                } else {
                    dfacc2_add(o.r, rh, rl, h[k].r.s, h[k].r.e);
                    dfacc2_add(o.i, rh, rl, h[k].i.s, h[k].i.e);
                }
                dfacc2_add(o.r, f2_neg(ih), f2_neg(il), h[k].i.s, h[k].i.e);
                dfacc2_add(o.i, ih, il, h[k].r.s, h[k].r.e);
            }
            if (nu == 3) {
                const df e0 = fwd ? emu : emum;
                const float2 ch = f2_dup(flip ? -e0.hi : e0.hi), cl = f2_dup(flip ? -e0.lo : e0.lo);
                dfacc2 t;
                dfacc2_first(t, ch, cl, o.r.s, o.r.e);
                o.r = t;
                dfacc2_first(t, ch, cl, o.i.s, o.i.e);
                o.i = t;
            }
            dfacc2_add_signed(up[a].r, one, o.r.s, o.r.e);
            dfacc2_add_signed(up[a].i, one, o.i.s, o.i.e);
            if (im) {
                dfacc2_add_signed(lw[a].r, f2_neg(lsg), o.i.s, o.i.e);
                dfacc2_add_signed(lw[a].i, lsg, o.r.s, o.r.e);
            } else {
                dfacc2_add_signed(lw[a].r, lsg, o.r.s, o.r.e);
                dfacc2_add_signed(lw[a].i, lsg, o.i.s, o.i.e);
            }
        }
    }
    const RegenCoefDf* __restrict__ rc = q.rc + i;
    const float4 kb = __ldg(&rc->kb), cg = __ldg(&rc->cg), cc = __ldg(&rc->cc);
    float4* __restrict__ xn = reinterpret_cast<float4*>(q.r[(i + 1) % 3]);
    float4* __restrict__ y = reinterpret_cast<float4*>(q.y);
    cp_async_wait<0>();
    if (!own) return;
#pragma unroll
    for (int P = 0; P < 2; ++P) {
        const float4 cr = __ldg(P ? &rc->cl : &rc->cu);
        const float ks_ = P ? 1.f : -1.f;
        const float2 kh = f2_dup(ks_ * kb.x), kl = f2_dup(ks_ * kb.y);
        const float2 arh = f2_dup(cr.x), arl = f2_dup(cr.y), aih = f2_dup(cr.z), ail = f2_dup(cr.w);
        const float2 grh = f2_dup(cg.x), grl = f2_dup(cg.y), gih = f2_dup(cg.z), gil = f2_dup(cg.w);
        const float2 crh = f2_dup(cc.x), crl = f2_dup(cc.y), cih = f2_dup(cc.z), cil = f2_dup(cc.w);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const size_t e = (size_t)(P * 3 + a) * 2 * V + site;
            CAcc2 s = P ? lw[a] : up[a];
            s.r = dfacc2_value(s.r);
            s.i = dfacc2_value(s.i);
            const int c = (P * 3 + a) * 2;
            const float4 xr = ps[c * RD_T], xi = ps[(c + 1) * RD_T];
            const float2 xrh = make_float2(xr.x, xr.y), xrl = make_float2(xr.z, xr.w);
            const float2 xih = make_float2(xi.x, xi.y), xil = make_float2(xi.z, xi.w);
            CAcc2 z;
            dfacc2_first(z.r, kh, kl, s.r.s, s.r.e);
            dfacc2_first(z.i, kh, kl, s.i.s, s.i.e);
            dfacc2_add(z.r, arh, arl, xrh, xrl);
            dfacc2_add(z.i, arh, arl, xih, xil);
            dfacc2_add(z.r, f2_neg(aih), f2_neg(ail), xih, xil);
            dfacc2_add(z.i, aih, ail, xrh, xrl);
            if (i > 0) {
                const float4 mr = c < 9 ? us[c * RD_T] : __ldg(xm + e);
                const float4 mi = c + 1 < 9 ? us[(c + 1) * RD_T] : __ldg(xm + e + V);
                const float2 mrh = make_float2(mr.x, mr.y), mrl = make_float2(mr.z, mr.w);
                const float2 mih = make_float2(mi.x, mi.y), mil = make_float2(mi.z, mi.w);
                dfacc2_add(z.r, grh, grl, mrh, mrl);
                dfacc2_add(z.i, grh, grl, mih, mil);
                dfacc2_add(z.r, f2_neg(gih), f2_neg(gil), mih, mil);
                dfacc2_add(z.i, gih, gil, mrh, mrl);
            }
            const dfacc2 zr = dfacc2_value(z.r), zi = dfacc2_value(z.i);
            xn[e] = make_float4(zr.s.x, zr.s.y, zr.e.x, zr.e.y);
            xn[e + V] = make_float4(zi.s.x, zi.s.y, zi.e.x, zi.e.y);
            const float4 y0 = y[e], y1 = y[e + V];
            // c z summed by itself, then added to y: every rounding at the scale of y's low part stays in y
            // for the rest of the pass (over 480 steps they are its error), and this way there is one
            dfacc2 yr, yi, pr, pi;
            yr.s = make_float2(y0.x, y0.y), yr.e = make_float2(y0.z, y0.w);
            yi.s = make_float2(y1.x, y1.y), yi.e = make_float2(y1.z, y1.w);
            dfacc2_first(pr, crh, crl, zr.s, zr.e);
            dfacc2_first(pi, crh, crl, zi.s, zi.e);
            dfacc2_add(pr, f2_neg(cih), f2_neg(cil), zi.s, zi.e);
            dfacc2_add(pi, cih, cil, zr.s, zr.e);
            dfacc2_add_tight(yr, pr.s, pr.e);
            dfacc2_add_tight(yi, pi.s, pi.e);
            yr = dfacc2_value(yr);
            yi = dfacc2_value(yi);
            y[e] = make_float4(yr.s.x, yr.s.y, yr.e.x, yr.e.y);
            y[e + V] = make_float4(yi.s.x, yi.s.y, yi.e.x, yi.e.y);
        }
    }
}

// ---- FP64 regeneration: one block per 32-site tile of a sequence: warp h applies hop h
// (direction-uniform code) to the tile's sites, the eight partial sums meet in shared memory, and 256
// threads (site, part) finish the components.
template <int MINB>
__global__ void __launch_bounds__(8 * TT, MINB) k_b_regen(const BSeq* __restrict__ S, const int* __restrict__ tseq, int i,
                                                    HopCoef<double> hc) {
    using R = double;
    using VT = double2;
    extern __shared__ __align__(16) unsigned char smraw[];
    cx<R>(*dirpart)[TT][6] = reinterpret_cast<cx<R>(*)[TT][6]>(smraw);  // [8][TT][2 spins x 3 colours]
    __shared__ cx<R> cf[4];
    const BSeq& q = S[tseq[blockIdx.x]];  // set-up data, not written by the solve
    const KState* ks = q.ks;
    pdl_wait_and_release();
    if (ks->status || i + 1 >= ks->kused) return;
    if (threadIdx.x == 0) {
        const cx<double> ib = cdiv(mk(1.0, 0.0), d2c(q.beta[i]));
        cf[0] = (ib);
        cf[1] = (ib * d2c(q.alpha[i]));
        cf[2] = (i > 0 ? ib * d2c(q.gamma[i - 1]) : mk(0.0, 0.0));
        cf[3] = (d2c(q.cvec[i + 1]));
    }
    const int tile = blockIdx.x - q.tile0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const VT* ri = (const VT*)q.r[i % 3];
    const void* U = q.U64;
    {
        // warp wid: hop wid of the tile's 32 sites, kept as its half spinor
        const int i0 = tile * TT + lane;
        if (i0 < q.g.V) {
            const Coord c = site_coord(q.g, i0);
            const VT* const xs[1] = {ri};
            const HopCoef<R> hcs[1] = {hc};
            Half<R> hp[1];
            hop_half_uniform<LINK_F64, R, 1>(wid, q.g, c, i0, U, xs, hp, hcs);
#pragma unroll
            for (int c6 = 0; c6 < 6; ++c6) dirpart[wid][lane][c6] = hp[0].h[c6 / 3][c6 % 3];
        }
    }
    __syncthreads();
    // epilogue: 256 threads (site, part), components part and part + 8 (< 12)
    const int site = threadIdx.x >> 3, part = threadIdx.x & 7;
    const int ii = tile * TT + site;
    if (ii >= q.g.V) return;
    const VT* rm = (const VT*)q.r[(i + 2) % 3];
    VT* rn = (VT*)q.r[(i + 1) % 3];
    VT* y = (VT*)q.y;
#pragma unroll
    for (int c2 = 0; c2 < 2; ++c2) {
        const int c = part + 8 * c2;
        if (c >= 12) break;
        const cx<R> self = ld_comp_cg<R>(ri, q.g.V, ii, c);
        cx<R> z = self;
        const int sp = c / 3, a = c % 3;
#pragma unroll
        for (int w = 0; w < 8; ++w) z = add_lazy(z, hop_spin<R>(w, sp, dirpart[w][site][a], dirpart[w][site][3 + a]));
        if (c >= 6) z = -z;  // gamma5: spins 2, 3
        z = mk(cf[0].r * z.r, cf[0].r * z.i) - cf[1] * self;  // 1 / beta_i is real
        if (i > 0) z = z - cf[2] * ld_comp_cg<R>(rm, q.g.V, ii, c);
        st_comp<R>(rn, q.g.V, ii, c, z);
        st_comp<R>(y, q.g.V, ii, c, ld_comp_cg<R>(y, q.g.V, ii, c) + cf[3] * z);
    }
}

// The regeneration step for two sequences of the same lattice per block (work entry: the two
// sequences, the tile, whether the second one exists): each hop warp loads the link and computes
// the neighbour index once and runs the two sequences' FP64 products as independent chains
// (twice the work in flight per warp); the epilogue spreads the 2 x 32 sites x 12 components over
// the 256 threads, three each.  Same arithmetic per sequence as k_b_regen.
template <int MINB>
__global__ void __launch_bounds__(8 * TT, MINB) k_b_regen2(const BSeq* __restrict__ S, const int4* __restrict__ work,
                                                     int i, HopCoef<double> hc) {
    using R = double;
    using VT = double2;
    extern __shared__ __align__(16) unsigned char smraw[];
    cx<R>(*dirpart)[8][TT][6] = reinterpret_cast<cx<R>(*)[8][TT][6]>(smraw);  // [2][8][TT][6]
    __shared__ cx<R> cf[2][4];
    const int4 wk = work[blockIdx.x];  // set-up data, not written by the solve
    const BSeq& qa = S[wk.x];
    const BSeq& qb = S[wk.y];
    const bool two = wk.w != 0;
    pdl_wait_and_release();
    const bool la = !(qa.ks->status || i + 1 >= qa.ks->kused);
    const bool lb = two && !(qb.ks->status || i + 1 >= qb.ks->kused);
    if (!la && !lb) return;
    if (threadIdx.x < 2 && (threadIdx.x == 0 || two)) {
        const BSeq& q = threadIdx.x ? qb : qa;
        const cx<double> ib = cdiv(mk(1.0, 0.0), d2c(q.beta[i]));
        cf[threadIdx.x][0] = (ib);
        cf[threadIdx.x][1] = (ib * d2c(q.alpha[i]));
        cf[threadIdx.x][2] = (i > 0 ? ib * d2c(q.gamma[i - 1]) : mk(0.0, 0.0));
        cf[threadIdx.x][3] = (d2c(q.cvec[i + 1]));
    }
    const int tile = wk.z;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const Geom& g = qa.g;
    const VT* ra = (const VT*)qa.r[i % 3];
    const VT* rb = two ? (const VT*)qb.r[i % 3] : ra;
    const void* U = qa.U64;
    {
        const int i0 = tile * TT + lane;
        if (i0 < g.V) {
            const Coord c = site_coord(g, i0);
            const VT* const xs[2] = {ra, rb};
            const HopCoef<R> hcs[2] = {hc, hc};
            Half<R> hp[2];
            hop_half_uniform<LINK_F64, R, 2>(wid, g, c, i0, U, xs, hp, hcs);
#pragma unroll
            for (int c6 = 0; c6 < 6; ++c6) {
                dirpart[0][wid][lane][c6] = hp[0].h[c6 / 3][c6 % 3];
                dirpart[1][wid][lane][c6] = hp[1].h[c6 / 3][c6 % 3];
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int rr = 0; rr < 3; ++rr) {
        const int task = threadIdx.x + rr * 8 * TT;
        const int sq = task / (TT * 12), rem = task % (TT * 12);
        const int site = rem / 12, c = rem % 12;
        if (sq ? !lb : !la) continue;
        const BSeq& q = sq ? qb : qa;
        const int ii = tile * TT + site;
        if (ii >= g.V) continue;
        const VT* ri = sq ? rb : ra;
        const VT* rm = (const VT*)q.r[(i + 2) % 3];
        VT* rn = (VT*)q.r[(i + 1) % 3];
        VT* y = (VT*)q.y;
        const cx<R> self = ld_comp_cg<R>(ri, g.V, ii, c);
        cx<R> z = self;
        const int sp = c / 3, a = c % 3;
#pragma unroll
        for (int w = 0; w < 8; ++w)
            z = add_lazy(z, hop_spin<R>(w, sp, dirpart[sq][w][site][a], dirpart[sq][w][site][3 + a]));
        if (c >= 6) z = -z;  // gamma5: spins 2, 3
        z = mk(cf[sq][0].r * z.r, cf[sq][0].r * z.i) - cf[sq][1] * self;  // 1 / beta_i is real
        if (i > 0) z = z - cf[sq][2] * ld_comp_cg<R>(rm, g.V, ii, c);
        st_comp<R>(rn, g.V, ii, c, z);
        st_comp<R>(y, g.V, ii, c, ld_comp_cg<R>(y, g.V, ii, c) + cf[sq][3] * z);
    }
}

}  // namespace
}  // namespace ovl

// ------------------------------------------------------------------ host side --
struct ovl_batch {
    std::vector<ovl_ctx*> ctx;
    std::vector<int> nrhs;
    std::vector<int> seq_ctx;   // context of each sequence
    int nseq = 0;
    int kcap = 0;
    int mode = -1;              // 1 mixed, 0 FP64 one pass (basis stored), 2 FP64 two pass
    cudaStream_t st = nullptr;
    cudaStream_t cap_st = nullptr;
    // device memory
    void* mem = nullptr;
    size_t mem_bytes = 0;
    ovl::BSeq* dseq = nullptr;
    int* dbseq[ovl::NSHAPE] = {nullptr, nullptr, nullptr};
    int* dtseq = nullptr;
    int4* dpair = nullptr;         // FP64 regeneration, two sequences per block: (a, b, tile, two)
    int npair_blocks = 0;
    int2* drd = nullptr;           // double-float regeneration work: (sequence, first site)
    int nrd = 0;
    unsigned int* pbar = nullptr;  // per-sequence barrier counters of the persistent pass 1
    int bp1_fit = -1;              // persistent pass 1 fits the GPU (-1: not yet determined)
    int nblocks[ovl::NSHAPE] = {0, 0, 0};
    int ntiles = 0;
    // autotuned launch shapes: pass-1 site-block shape, blocks per SM of the regeneration kernel
    int shape = 1;
    int regen_minb = 3;
    int regen_pair = 0;         // 1: two sequences of one lattice per regeneration block
    bool tuned = false;
    bool pinned = false;        // shapes set by ovl_batch_set_tuning: never retuned
    bool tune_cached = false;   // the shapes came from the tuning cache (no timing)
    int tuned_kind = -1;        // tune_kind of the shapes
    std::vector<ovl::BSeq> hseq;
    std::vector<double2*> b64, bR, bL, pq;
    ovl::KState* ks = nullptr;
    double2 *alpha = nullptr, *beta = nullptr, *gamma = nullptr, *cvec = nullptr, *vscale = nullptr;
    double2* inner = nullptr;
    size_t inner_stride = 0;
    double* qpart = nullptr;
    size_t qpart_stride = 0;
    unsigned int* qcnt = nullptr;
    double* part = nullptr;      // scratch of the per-sequence prologue kernels (pro_off[s] doubles in)
    std::vector<size_t> pro_off;
    std::vector<int> pro_m;      // deflation sizes the prologue scratch was laid out for
    unsigned int* counter = nullptr;
    // the sequences' prologues run on side streams (graph branches), joined before pass 1
    static constexpr int NSIDE = 4;
    cudaStream_t side[NSIDE] = {nullptr, nullptr, nullptr, nullptr};
    cudaEvent_t ev_fork = nullptr;
    cudaEvent_t ev_join[NSIDE] = {nullptr, nullptr, nullptr, nullptr};
    double2* stage = nullptr;    // host transfers
    // per-phase profile (OVL_PROFILE): pass 1, inner sign, pass 2 / combination
    double prof_ms[3] = {0.0, 0.0, 0.0};
    int prof_n = 0;
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
    // graph
    cudaGraphExec_t exec = nullptr;
    int g_k = -1, g_flags = 0;
    std::vector<int> g_m;  // deflation size of every context when the graph was captured
    double g_mu = 0, g_kappa = 0;
    std::string err;
};

namespace {

int bfail(ovl_batch* b, int code, const std::string& m) {
    if (b) b->err = m;
    return code;
}

void bfree(ovl_batch* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
    if (b->mem) cudaFree(b->mem);
    b->mem = nullptr;
    b->mem_bytes = 0;
    b->mode = -1;
}

// Carve the batch's device memory for mode (1 mixed, 0 FP64 one pass, 2 FP64 two pass) and Krylov size kmax.
int balloc(ovl_batch* b, int mode, int kmax) {
    if (b->mem && b->mode == mode && b->kcap >= kmax) return OVL_OK;
    bfree(b);
    const int ns = b->nseq;
    const size_t kk = (size_t)kmax + 2;
    const size_t inner_stride = std::max(ovl::inner_work_elems(kmax, 0), ovl::inner_work_elems(kmax, 1));
    const size_t qpart_stride = 8192;
    // byte sizes, every piece 256-aligned
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    size_t total = 0;
    std::vector<size_t> seq_bytes(ns);
    int nblocks[ovl::NSHAPE] = {0, 0, 0}, ntiles = 0;
    for (int s = 0; s < ns; ++s) {
        const ovl_ctx* c = b->ctx[b->seq_ctx[s]];
        const size_t n = c->n;
        // partials: the most blocks of a pass-1 shape, or two sets for the persistent pass 1
        const int nblk = std::max((c->g.V + ovl::SHAPE_SITES[0] - 1) / ovl::SHAPE_SITES[0],
                                  2 * ((c->g.V + ovl::BP1_T - 1) / ovl::BP1_T));
        for (int h = 0; h < ovl::NSHAPE; ++h) nblocks[h] += (c->g.V + ovl::SHAPE_SITES[h] - 1) / ovl::SHAPE_SITES[h];
        ntiles += (c->g.V + ovl::TT - 1) / ovl::TT;
        size_t z = 0;
        z += 4 * al(n * sizeof(double2));                        // b, bR, bL, y
        z += 3 * al(n * sizeof(double2));                        // regeneration ring
        if (mode == 1) z += 8 * al(n * sizeof(float2));          // FP32 v, w rings, t, s
        else if (mode == 0) z += (kk + 5) * al(n * sizeof(double2));  // FP64 basis, w ring, t, s
        else z += 8 * al(n * sizeof(double2));                  // FP64 v, w rings, t, s
        z += al((size_t)nblk * 4 * sizeof(double2)) + al(128 * sizeof(double2));  // partials, pq
        seq_bytes[s] = z;
        total += z;
    }
    // prologue scratch per sequence: the two-stage projections' partials (m vectors x blocks,
    // complex) or the deflation split's grid sum (4 values x at most 512 blocks)
    // two sequences of one lattice per regeneration block (the sources of a context are consecutive)
    std::vector<int4> ptable;
    {
        int s0 = 0;
        for (size_t j = 0; j < b->ctx.size(); ++j) {
            const int nt = (b->ctx[j]->g.V + ovl::TT - 1) / ovl::TT;
            for (int r = 0; r < b->nrhs[j]; r += 2) {
                const int sa = s0 + r, two = r + 1 < b->nrhs[j];
                const int sb = two ? sa + 1 : sa;
                for (int t = 0; t < nt; ++t) ptable.push_back(make_int4(sa, sb, t, two));
            }
            s0 += b->nrhs[j];
        }
    }
    // double-float regeneration: blocks of RD_T sites of one sequence, a lattice's sequences side by
    // side (the same links are read at about the same time)
    std::vector<int2> rtable;
    if (mode == 1) {
        int s0 = 0;
        for (size_t j = 0; j < b->ctx.size(); ++j) {
            for (int site = 0; site < b->ctx[j]->g.V; site += ovl::RD_T)
                for (int r = 0; r < b->nrhs[j]; ++r) rtable.push_back(make_int2(s0 + r, site));
            s0 += b->nrhs[j];
        }
    }
    const size_t rcb = mode == 1 ? ns * kk * sizeof(ovl::RegenCoefDf) : 0;
    std::vector<size_t> pro_off(ns + 1, 0);
    std::vector<int> pro_m(ns, 0);
    for (int s = 0; s < ns; ++s) {
        const ovl_ctx* c = b->ctx[b->seq_ctx[s]];
        pro_m[s] = c->m;
        const size_t need = std::max<size_t>((size_t)2 * std::max(c->m, 1) * ovl::multidot_blocks(c->n), 2048);
        pro_off[s + 1] = pro_off[s] + ((need + 31) & ~(size_t)31);
    }
    total += al(ns * sizeof(ovl::KState)) + 5 * al(ns * kk * sizeof(double2)) + al(ns * 4 * sizeof(double2)) +
             al((size_t)ns * inner_stride * sizeof(double2)) + al((size_t)ns * qpart_stride * sizeof(double)) +
             al(ns * 64 * sizeof(unsigned int)) + al(ns * sizeof(ovl::BSeq)) + al(nblocks[0] * sizeof(int)) +
             al(nblocks[1] * sizeof(int)) + al(nblocks[2] * sizeof(int)) +
             al(ntiles * sizeof(int)) + al(ns * sizeof(unsigned int)) + al(ptable.size() * sizeof(int4)) +
             al(rtable.size() * sizeof(int2)) + al(rcb) +
             al(pro_off[ns] * sizeof(double)) + al(64 * sizeof(unsigned int));
    if (cudaMalloc(&b->mem, total) != cudaSuccess) {
        b->mem = nullptr;
        return bfail(b, OVL_ENOMEM, "batch workspace");
    }
    b->mem_bytes = total;
    char* p = (char*)b->mem;
    auto take = [&](size_t bytes) { char* r = p; p += al(bytes); return (void*)r; };
    b->ks = (ovl::KState*)take(ns * sizeof(ovl::KState));
    b->alpha = (double2*)take(ns * kk * sizeof(double2));
    b->beta = (double2*)take(ns * kk * sizeof(double2));
    b->gamma = (double2*)take(ns * kk * sizeof(double2));
    b->cvec = (double2*)take(ns * kk * sizeof(double2));
    b->vscale = (double2*)take(ns * kk * sizeof(double2));
    double2* cf = (double2*)take(ns * 4 * sizeof(double2));
    b->inner = (double2*)take((size_t)ns * inner_stride * sizeof(double2));
    b->inner_stride = inner_stride;
    b->qpart = (double*)take((size_t)ns * qpart_stride * sizeof(double));
    b->qpart_stride = qpart_stride;
    b->qcnt = (unsigned int*)take(ns * 64 * sizeof(unsigned int));
    b->dseq = (ovl::BSeq*)take(ns * sizeof(ovl::BSeq));
    for (int h = 0; h < ovl::NSHAPE; ++h) b->dbseq[h] = (int*)take(nblocks[h] * sizeof(int));
    b->dtseq = (int*)take(ntiles * sizeof(int));
    b->pbar = (unsigned int*)take(ns * sizeof(unsigned int));
    b->dpair = (int4*)take(ptable.size() * sizeof(int4));
    b->npair_blocks = (int)ptable.size();
    b->drd = (int2*)take(rtable.size() * sizeof(int2));
    b->nrd = (int)rtable.size();
    ovl::RegenCoefDf* rc = (ovl::RegenCoefDf*)take(rcb);
    b->part = (double*)take(pro_off[ns] * sizeof(double));
    b->pro_off = pro_off;
    b->pro_m = pro_m;
    b->counter = (unsigned int*)take(64 * sizeof(unsigned int));
    b->hseq.assign(ns, ovl::BSeq());
    b->b64.assign(ns, nullptr), b->bR.assign(ns, nullptr), b->bL.assign(ns, nullptr), b->pq.assign(ns, nullptr);
    std::vector<int> table[ovl::NSHAPE], ttable;
    ttable.reserve(ntiles);
    int blk0[ovl::NSHAPE] = {0, 0, 0}, tile0 = 0;
    for (int s = 0; s < ns; ++s) {
        ovl_ctx* c = b->ctx[b->seq_ctx[s]];
        const size_t n = c->n;
        ovl::BSeq& q = b->hseq[s];
        std::memset(&q, 0, sizeof(q));
        q.g = c->g;
        q.n = n;
        q.U = mode == 1 ? (const void*)c->U12 : (const void*)c->U64;
        q.U64 = c->U64;
        q.Udf = c->Udf;
        q.nbr = c->nbr;
        b->b64[s] = (double2*)take(n * sizeof(double2));
        b->bR[s] = (double2*)take(n * sizeof(double2));
        b->bL[s] = (double2*)take(n * sizeof(double2));
        q.y = (double2*)take(n * sizeof(double2));
        q.bR = b->bR[s];
        q.rc = mode == 1 ? rc + s * kk : nullptr;
        for (int j = 0; j < 3; ++j) q.r[j] = (double2*)take(n * sizeof(double2));
        if (mode == 1) {
            for (int j = 0; j < 3; ++j) q.v[j] = take(n * sizeof(float2)), q.w[j] = take(n * sizeof(float2));
            q.t = take(n * sizeof(float2));
            q.s = take(n * sizeof(float2));
            q.V = nullptr;
        } else if (mode == 0) {
            q.V = (double2*)take(kk * n * sizeof(double2));
            for (int j = 0; j < 3; ++j) q.w[j] = take(n * sizeof(double2)), q.v[j] = nullptr;
            q.t = take(n * sizeof(double2));
            q.s = take(n * sizeof(double2));
        } else {
            for (int j = 0; j < 3; ++j) q.v[j] = take(n * sizeof(double2)), q.w[j] = take(n * sizeof(double2));
            q.t = take(n * sizeof(double2));
            q.s = take(n * sizeof(double2));
            q.V = nullptr;
        }
        q.ks = b->ks + s;
        q.alpha = b->alpha + s * kk;
        q.beta = b->beta + s * kk;
        q.gamma = b->gamma + s * kk;
        q.cvec = b->cvec + s * kk;
        q.vscale = b->vscale + s * kk;
        q.cf = cf + 4 * s;
        for (int h = 0; h < ovl::NSHAPE; ++h) q.nblk[h] = (c->g.V + ovl::SHAPE_SITES[h] - 1) / ovl::SHAPE_SITES[h];
        q.part = (double2*)take((size_t)std::max(q.nblk[0], 2 * q.nblk[1]) * 4 * sizeof(double2));
        b->pq[s] = (double2*)take(128 * sizeof(double2));
        q.cnt = b->qcnt + s;  // the inner quadrature's counters follow at qcnt + nseq
        for (int h = 0; h < ovl::NSHAPE; ++h) {
            q.blk0[h] = blk0[h];
            for (int j = 0; j < q.nblk[h]; ++j) table[h].push_back(s);
            blk0[h] += q.nblk[h];
        }
        q.ntile = (c->g.V + ovl::TT - 1) / ovl::TT;
        q.tile0 = tile0;
        for (int j = 0; j < q.ntile; ++j) ttable.push_back(s);
        tile0 += q.ntile;
    }
    for (int h = 0; h < ovl::NSHAPE; ++h) b->nblocks[h] = blk0[h];
    b->ntiles = tile0;
    if (cudaMemcpy(b->dseq, b->hseq.data(), ns * sizeof(ovl::BSeq), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->dbseq[0], table[0].data(), table[0].size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->dbseq[1], table[1].data(), table[1].size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->dbseq[2], table[2].data(), table[2].size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->dtseq, ttable.data(), ttable.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->dpair, ptable.data(), ptable.size() * sizeof(int4), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->drd, rtable.data(), rtable.size() * sizeof(int2), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(b->qcnt, 0, ns * 64 * sizeof(unsigned int)) != cudaSuccess ||
        cudaMemset(b->counter, 0, 64 * sizeof(unsigned int)) != cudaSuccess) {
        bfree(b);
        return bfail(b, OVL_ECUDA, "batch set-up copies");
    }
    b->mode = mode;
    b->kcap = kmax;
    return OVL_OK;
}

// Launch with programmatic stream serialisation (see pdl_wait_and_release).
template <typename... KArgs, typename... Args>
void launch_pdl(void (*kern)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, args...);
}

// The whole FP32 pass 1 as one cooperative launch when all of the batch's sites fit the GPU at once.
bool bp1_fits(ovl_batch* b) {
    if (b->bp1_fit < 0) {
        int per_sm = 0, nsm = 0, dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ovl::k_bp1<ovl::LINK_F32_12>, ovl::BP1_T, 0);
        b->bp1_fit = (per_sm > 0 && b->nblocks[1] <= per_sm * nsm) ? 1 : 0;
    }
    return b->bp1_fit == 1;
}

int launch_bp1(ovl_batch* b, int k, double mu, double kappa, cudaStream_t st) {
    if (cudaMemsetAsync(b->pbar, 0, b->nseq * sizeof(unsigned int), st) != cudaSuccess) return OVL_ECUDA;
    ovl::BP1Args a;
    a.S = b->dseq;
    a.bseq = b->dbseq[1];
    a.bar = b->pbar;
    a.k = k;
    a.hv = ovl::make_coef<float>(mu, kappa);
    a.hw = ovl::make_coef<float>(-mu, kappa);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b->nblocks[1]);
    cfg.blockDim = dim3(ovl::BP1_T);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, ovl::k_bp1<ovl::LINK_F32_12>, a) == cudaSuccess ? OVL_OK : OVL_ECUDA;
}

// One pass-1 step of every sequence with site-block shape SH.
template <int SH>
void pass1_step(ovl_batch* b, int i, int k, double mu, double kappa, bool mixed, cudaStream_t st) {
    const int nb = b->nblocks[SH], T = ovl::SHAPE_SITES[SH];
    const ovl::BSeq* S = b->dseq;
    const int* tab = b->dbseq[SH];
    if (mixed) {
        launch_pdl(ovl::k_b_pair<ovl::LINK_F32_12, float, SH>, dim3(nb, 2), T, 0, st, S, tab, i, k - 1,
                   ovl::make_coef<float>(mu, kappa), ovl::make_coef<float>(-mu, kappa));
        if (i + 1 < k) launch_pdl(ovl::k_b_lstep<float, SH>, nb, T, 0, st, S, tab, i);
    } else {
        launch_pdl(ovl::k_b_pair<ovl::LINK_F64, double, SH>, dim3(nb, 2), T, 0, st, S, tab, i, k - 1,
                   ovl::make_coef<double>(mu, kappa), ovl::make_coef<double>(-mu, kappa));
        if (i + 1 < k) launch_pdl(ovl::k_b_lstep<double, SH>, nb, T, 0, st, S, tab, i);
    }
}

// One double-float regeneration step of every sequence, compiled for 3 or 4 times 128 threads per SM (163
// or 128 registers).  Neither is best everywhere: 48 sequences on four lattices 303 / 290 us, 12 on 8^4
// 28.9 / 36.8 us (768 blocks: at eight per SM the next step's blocks, launched early, crowd on a few SMs).
template <int MINB>
void regen_df_step(ovl_batch* b, int i, double mu, cudaStream_t st) {
    static unsigned long long attr_dev = 0;
    if (ovl::first_use_on_device(attr_dev))
        cudaFuncSetAttribute(ovl::k_b_regen_df<MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ovl::RD_SM);
    launch_pdl(ovl::k_b_regen_df<MINB>, b->nrd, ovl::RD_T, ovl::RD_SM, st, (const ovl::BSeq*)b->dseq,
               (const int2*)b->drd, i, ovl::df(exp(mu)), ovl::df(exp(-mu)));
}

// One FP64 regeneration step of every sequence, blocks-per-SM bound MINB (one or two sequences per block).
template <int MINB>
void regen_step(ovl_batch* b, int i, double mu, double kappa, cudaStream_t st) {
    const ovl::BSeq* S = b->dseq;
    const size_t smr = (size_t)8 * ovl::TT * 6 * 16;
    static unsigned long long attr_dev = 0;
    if (ovl::first_use_on_device(attr_dev)) {
        cudaFuncSetAttribute(ovl::k_b_regen<MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smr);
        cudaFuncSetAttribute(ovl::k_b_regen2<MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(2 * smr));
    }
    if (b->regen_pair)
        launch_pdl(ovl::k_b_regen2<MINB>, b->npair_blocks, 8 * ovl::TT, 2 * smr, st, S, (const int4*)b->dpair, i,
                   ovl::make_coef<double>(mu, kappa));
    else
        launch_pdl(ovl::k_b_regen<MINB>, b->ntiles, 8 * ovl::TT, smr, st, S, (const int*)b->dtseq, i,
                   ovl::make_coef<double>(mu, kappa));
}

// Everything between the packed sources and the unpacked results, on stream st.
int enqueue_batch(ovl_batch* b, int k, double mu, double kappa, int flags, cudaStream_t st) {
    if (k > b->kcap) return bfail(b, OVL_EINVAL, "k exceeds the batch workspace");
    const bool mixed = b->mode == 1;
    const bool twopass = b->mode != 0;
    const int ns = b->nseq;
    const bool prof = (flags & OVL_PROFILE) != 0;
    // prologue of every sequence (deflation split, start vectors): independent, so they run on
    // side streams forked from st and joined before pass 1 (parallel branches of the graph)
    const int nside = std::min(ns, ovl_batch::NSIDE);
    if (!b->ev_fork) {
        if (cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming) != cudaSuccess)
            return bfail(b, OVL_ECUDA, "prologue events");
        for (int j = 0; j < ovl_batch::NSIDE; ++j)
            if (cudaStreamCreateWithFlags(&b->side[j], cudaStreamNonBlocking) != cudaSuccess ||
                cudaEventCreateWithFlags(&b->ev_join[j], cudaEventDisableTiming) != cudaSuccess)
                return bfail(b, OVL_ECUDA, "prologue streams");
    }
    cudaEventRecord(b->ev_fork, st);
    for (int j = 0; j < nside; ++j) cudaStreamWaitEvent(b->side[j], b->ev_fork, 0);
    for (int s = 0; s < ns; ++s) {
        cudaStream_t ss = b->side[s % nside];
        ovl_ctx* c = b->ctx[b->seq_ctx[s]];
        const ovl::BSeq& q = b->hseq[s];
        const size_t n = q.n;
        double* part = b->part + b->pro_off[s];
        unsigned int* cnt = b->qcnt + 2 * ns + s;  // zero between uses (the last block resets it)
        ovl::launch_state_init(q.ks, ss);
        const int m = c->m;
        if (m > 0) {
            ovl::launch_multidot(c->L, n, m, b->b64[s], b->pq[s], 0, part, n, ss);
            ovl::launch_multidot(c->R, n, m, b->b64[s], b->pq[s] + m, 0, part, n, ss);
        }
        ovl::launch_deflate_split(b->b64[s], c->R, c->L, c->lam, m, b->pq[s], b->bR[s], b->bL[s], q.y, q.ks,
                                  q.vscale, part, cnt, n, ss);
        if (mixed) {
            ovl::launch_native_f64_to_f32(b->bR[s], q.v[0], q.g, 1, ss);
            ovl::launch_native_f64_to_f32(b->bL[s], q.w[0], q.g, 1, ss);
        } else {
            cudaMemcpyAsync(q.V ? (void*)q.V : q.v[0], b->bR[s], n * sizeof(double2), cudaMemcpyDeviceToDevice, ss);
            cudaMemcpyAsync(q.w[0], b->bL[s], n * sizeof(double2), cudaMemcpyDeviceToDevice, ss);
        }
    }
    for (int j = 0; j < nside; ++j) {
        cudaEventRecord(b->ev_join[j], b->side[j]);
        cudaStreamWaitEvent(st, b->ev_join[j], 0);
    }
    // pass 1 (all sequences per launch): one persistent launch for mixed batches that fit the GPU
    if (prof) cudaEventRecord(b->ev[0], st);
    if (mixed && !(flags & OVL_STEPWISE) && bp1_fits(b)) {
        if (launch_bp1(b, k, mu, kappa, st)) return bfail(b, OVL_ECUDA, "persistent pass-1 launch");
    } else
    for (int i = 0; i < k; ++i) {
        switch (b->shape) {
            case 0: pass1_step<0>(b, i, k, mu, kappa, mixed, st); break;
            case 1: pass1_step<1>(b, i, k, mu, kappa, mixed, st); break;
            default: pass1_step<2>(b, i, k, mu, kappa, mixed, st); break;
        }
    }
    // inner sign of every sequence at once; Roberts' iteration where the quadrature did not settle
    if (prof) cudaEventRecord(b->ev[1], st);
    const size_t kk = (size_t)b->kcap + 2;
    if (ovl::launch_inner_quadrature_batched(ns, b->alpha, b->beta, b->gamma, b->ks, b->cvec, kk, b->inner,
                                             b->inner_stride, b->kcap, b->qpart, b->qpart_stride, b->qcnt + ns, st))
        return bfail(b, OVL_ECUDA, "batched inner sign launch");
    for (int s = 0; s < ns; ++s) {
        ovl_ctx* c = b->ctx[b->seq_ctx[s]];
        const ovl::BSeq& q = b->hseq[s];
        if (ovl::launch_inner_newton(q.alpha, q.beta, q.gamma, nullptr, 0, 1, q.ks, q.cvec,
                                     b->inner + (size_t)s * b->inner_stride, b->inner_stride, b->kcap, c->num_sms, st,
                                     1))
            return bfail(b, OVL_ECUDA, "inner sign fallback launch");
    }
    // combination
    if (prof) cudaEventRecord(b->ev[2], st);
    if (twopass) {
        // mixed: double-float regeneration unless OVL_PASS2_F64 (ring and y converted in place)
        const bool dfm = mixed && !(flags & OVL_PASS2_F64);
        if (dfm) {
            if (k > 1) ovl::k_b_regen_coef<<<dim3((k + 126) / 128, ns), 128, 0, st>>>(b->dseq, kappa);
            ovl::k_b_regen_start<<<b->nblocks[1], 128, 0, st>>>(b->dseq, b->dbseq[1]);
        } else {
            for (int s = 0; s < ns; ++s) {
                const ovl::BSeq& q = b->hseq[s];
                ovl::launch_scale_start(b->bR[s], q.r[0], q.y, q.cvec, q.ks, q.n, st);
            }
        }
        for (int i = 0; i + 1 < k; ++i) {
            if (dfm) {
                if (b->regen_minb <= 3) regen_df_step<3>(b, i, mu, st);
                else regen_df_step<4>(b, i, mu, st);
                continue;
            }
            switch (b->regen_minb) {
                case 2: regen_step<2>(b, i, mu, kappa, st); break;
                case 4: regen_step<4>(b, i, mu, kappa, st); break;
                case 5: regen_step<5>(b, i, mu, kappa, st); break;
                case 6: regen_step<6>(b, i, mu, kappa, st); break;
                default: regen_step<3>(b, i, mu, kappa, st); break;
            }
        }
        if (dfm) ovl::k_b_regen_out<<<b->nblocks[1], 128, 0, st>>>(b->dseq, b->dbseq[1]);
    } else {
        for (int s = 0; s < ns; ++s) {
            const ovl::BSeq& q = b->hseq[s];
            ovl::launch_combine(q.V, q.n, q.vscale, q.cvec, q.ks, b->kcap, q.y, q.n, st);
        }
    }
    if (prof) cudaEventRecord(b->ev[3], st);
    return cudaGetLastError() == cudaSuccess ? OVL_OK : bfail(b, OVL_ECUDA, "batch launch");
}

// Tuning cache: the chosen shapes per (GPU model, SM count, precision, lattice extents and
// right-hand sides of every context), kept for the process and, when the environment variable
// OVL_TUNE_CACHE names a file, in that file ("key shape minb pair" per line) across processes.
std::mutex g_tune_mu;
std::map<std::string, std::array<int, 3>> g_tune;

// What the tuned shapes were timed with: the workspace mode, and in the mixed one which regeneration runs
// (mode 3: the FP64 kernels of OVL_PASS2_F64, whose candidates and best shapes are others).
int tune_kind(const ovl_batch* b, int flags) { return b->mode == 1 && (flags & OVL_PASS2_F64) ? 3 : b->mode; }

std::string tune_key(const ovl_batch* b, int kind) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceProp pr{};
    cudaGetDeviceProperties(&pr, dev);
    // ("/r3": the double-float regeneration of one thread per site, and the FP64 one under a key of its own;
    // lines of other forms do not apply)
    std::string k = std::string(pr.name) + "/" + std::to_string(pr.multiProcessorCount) + "/r3/m" + std::to_string(kind);
    for (size_t j = 0; j < b->ctx.size(); ++j) {
        const ovl::Geom& g = b->ctx[j]->g;
        k += "/" + std::to_string(g.L[0]) + "x" + std::to_string(g.L[1]) + "x" + std::to_string(g.L[2]) + "x" +
             std::to_string(g.L[3]) + "r" + std::to_string(b->nrhs[j]);
    }
    for (char& ch : k)
        if (ch == ' ') ch = '_';
    return k;
}

bool tune_lookup(const std::string& key, std::array<int, 3>& out) {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune.find(key);
    if (it == g_tune.end()) {
        const char* path = std::getenv("OVL_TUNE_CACHE");
        if (path && *path) {
            std::ifstream f(path);
            std::string kk;
            int a, m, q;
            while (f >> kk >> a >> m >> q) g_tune[kk] = {a, m, q};
        }
        it = g_tune.find(key);
        if (it == g_tune.end()) return false;
    }
    out = it->second;
    return out[0] >= 0 && out[0] < ovl::NSHAPE && out[1] >= 2 && out[1] <= 6 && (out[2] == 0 || out[2] == 1);
}

void tune_store(const std::string& key, const std::array<int, 3>& v) {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune[key] = v;
    const char* path = std::getenv("OVL_TUNE_CACHE");
    if (path && *path) {
        std::ofstream f(path, std::ios::app);
        f << key << " " << v[0] << " " << v[1] << " " << v[2] << "\n";
    }
}

// Autotuner of the batched kernels' launch shapes (site-block size of the pass-1 kernels, blocks
// per SM of the regeneration kernel): each candidate runs a short eager solve (TUNE_K steps) of the
// whole batch with events around its phases; the fastest pass-1 and regeneration candidates are
// kept for the batch.  The sources must already be packed.  fixed_shape >= 0: pass 1 keeps that shape.
int autotune(ovl_batch* b, double mu, double kappa, int flags, int fixed_shape, cudaStream_t st) {
    if (b->kcap < 8) return OVL_OK;  // too short to time; the defaults stay until a longer solve
    const int TUNE_K = std::min(24, b->kcap);  // the workspace holds kcap steps
    const int saved_shape = b->shape, saved_minb = b->regen_minb;
    for (cudaEvent_t& e : b->ev)
        if (!e && cudaEventCreate(&e) != cudaSuccess) return bfail(b, OVL_ECUDA, "tuning events");
    // candidates: pass-1 site-block shape, regeneration blocks per SM, sequences per regeneration block
    struct Cand {
        int shape, minb, pair;
    };
    // the double-float regeneration has two forms (3 or 4 times 128 threads per SM), the FP64 one seven
    const Cand cands[] = {{0, 3, 0}, {1, 4, 0}, {2, 5, 0}, {1, 6, 0}, {1, 2, 1}, {1, 3, 1}, {1, 4, 1}};
    const Cand cands_df[] = {{0, 3, 0}, {1, 4, 0}, {2, 4, 0}};
    const bool dfm = b->mode == 1 && !(flags & OVL_PASS2_F64);
    const Cand* cand = dfm ? cands_df : cands;
    const int ncand = dfm ? (int)(sizeof(cands_df) / sizeof(cands_df[0])) : (int)(sizeof(cands) / sizeof(cands[0]));
    float best1 = 1e30f, best2 = 1e30f;
    int bs = saved_shape, bm = saved_minb, bp = b->regen_pair;
    for (int rep = 0; rep < 2; ++rep)  // the first round warms caches and instruction memory
        for (int c = 0; c < ncand; ++c) {
            b->shape = cand[c].shape;
            b->regen_minb = cand[c].minb;
            b->regen_pair = cand[c].pair;
            const int r = enqueue_batch(b, TUNE_K, mu, kappa, (flags | OVL_PROFILE) & ~OVL_NO_GRAPH, st);
            if (r) return r;
            if (cudaStreamSynchronize(st) != cudaSuccess) return bfail(b, OVL_ECUDA, "tuning solve");
            float t1 = 0.f, t2 = 0.f;
            cudaEventElapsedTime(&t1, b->ev[0], b->ev[1]);
            cudaEventElapsedTime(&t2, b->ev[2], b->ev[3]);
            if (rep == 1) {
                if (t1 < best1) best1 = t1, bs = cand[c].shape;
                if (t2 < best2) best2 = t2, bm = cand[c].minb, bp = cand[c].pair;
            }
        }
    b->shape = fixed_shape >= 0 ? fixed_shape : bs;
    b->regen_minb = bm;
    b->regen_pair = bp;
    b->tuned = true;
    b->tuned_kind = tune_kind(b, flags);
    if (b->exec) cudaGraphExecDestroy(b->exec);  // a captured graph holds the old shapes
    b->exec = nullptr;
    return OVL_OK;
}

}  // namespace

extern "C" {

int ovl_batch_tuning(const ovl_batch* b, int* pass1_block_sites, int* regen_blocks_per_sm, int* regen_seqs_per_block) {
    if (!b) return OVL_EINVAL;
    if (pass1_block_sites) *pass1_block_sites = ovl::SHAPE_SITES[b->shape];
    if (regen_blocks_per_sm) *regen_blocks_per_sm = b->regen_minb;
    if (regen_seqs_per_block) *regen_seqs_per_block = b->regen_pair ? 2 : 1;
    return b->tuned ? OVL_OK : OVL_ESTATE;
}

int ovl_batch_set_tuning(ovl_batch* b, int pass1_block_sites, int regen_blocks_per_sm, int regen_seqs_per_block) {
    if (!b) return OVL_EINVAL;
    int sh = -1;
    for (int c = 0; c < ovl::NSHAPE; ++c)
        if (ovl::SHAPE_SITES[c] == pass1_block_sites) sh = c;
    if (sh < 0 || regen_blocks_per_sm < 2 || regen_blocks_per_sm > 6 || regen_seqs_per_block < 1 ||
        regen_seqs_per_block > 2)
        return bfail(b, OVL_EINVAL, "unsupported launch shape");
    b->shape = sh;
    b->regen_minb = regen_blocks_per_sm;
    b->regen_pair = regen_seqs_per_block == 2;
    b->tuned = b->pinned = true;
    if (b->exec) cudaGraphExecDestroy(b->exec);  // a captured graph holds the old shapes
    b->exec = nullptr;
    return OVL_OK;
}

int ovl_batch_create(ovl_batch** out, ovl_ctx* const* ctxs, int nctx, const int* nrhs) {
    if (!out || !ctxs || nctx < 1 || !nrhs) return OVL_EINVAL;
    *out = nullptr;
    ovl_batch* b = new ovl_batch();
    for (int j = 0; j < nctx; ++j) {
        if (!ctxs[j] || nrhs[j] < 0) {
            delete b;
            return OVL_EINVAL;
        }
        if (!ctxs[j]->have_gauge) {
            delete b;
            return OVL_ESTATE;
        }
        b->ctx.push_back(ctxs[j]);
        b->nrhs.push_back(nrhs[j]);
        for (int r = 0; r < nrhs[j]; ++r) b->seq_ctx.push_back(j);
    }
    b->nseq = (int)b->seq_ctx.size();
    if (b->nseq == 0) {
        delete b;
        return OVL_EINVAL;
    }
    b->st = ctxs[0]->st;
    *out = b;
    return OVL_OK;
}

int ovl_batch_destroy(ovl_batch* b) {
    if (!b) return OVL_OK;
    if (b->st) cudaStreamSynchronize(b->st);
    else cudaDeviceSynchronize();
    bfree(b);
    if (b->cap_st) cudaStreamDestroy(b->cap_st);
    for (cudaEvent_t e : b->ev)
        if (e) cudaEventDestroy(e);
    for (int j = 0; j < ovl_batch::NSIDE; ++j) {
        if (b->side[j]) cudaStreamDestroy(b->side[j]);
        if (b->ev_join[j]) cudaEventDestroy(b->ev_join[j]);
    }
    if (b->ev_fork) cudaEventDestroy(b->ev_fork);
    delete b;
    return OVL_OK;
}

const char* ovl_batch_last_error(const ovl_batch* b) { return b ? b->err.c_str() : "null batch"; }

int ovl_batch_solve(ovl_batch* b, int k, double mu, double kappa, const void* const* bsrc, void* const* out,
                    int flags, ovl_info* info) {
    if (!b || !bsrc || !out || k < 1) return bfail(b, OVL_EINVAL, "bad argument");
    // FP64: the basis is stored when it fits a fixed budget, else the regeneration pass is used
    size_t ntot = 0;
    for (int q = 0; q < b->nseq; ++q) ntot += b->ctx[b->seq_ctx[q]]->n;
    const bool fits = ((size_t)k + 2) * ntot * sizeof(double2) <= ((size_t)32 << 30);
    const int mode = (flags & OVL_MIXED) ? 1 : ((flags & OVL_TWO_PASS) || !fits) ? 2 : 0;
    // a deflation set larger than the prologue scratch was laid out for: lay the workspace out again
    if (b->mem)
        for (int q = 0; q < b->nseq; ++q)
            if (b->ctx[b->seq_ctx[q]]->m > b->pro_m[q]) {
                bfree(b);
                break;
            }
    int r = balloc(b, mode, k);
    if (r) return r;
    for (ovl_ctx* c : b->ctx) {
        if (c->m > 0 && mode == 1 && !c->R32) return bfail(b, OVL_ESTATE, "deflation set not installed");
        if (c->st != b->st) return bfail(b, OVL_EINVAL, "all contexts of a batch must share one stream");
    }
    cudaStream_t st = b->st;
    const bool host = (flags & OVL_HOST) != 0;
    // pack the sources (canonical -> device layout); sources of context j follow one another
    int s = 0;
    for (size_t j = 0; j < b->ctx.size(); ++j) {
        ovl_ctx* c = b->ctx[j];
        const size_t n = c->n, vb = n * sizeof(double2);
        for (int rr = 0; rr < b->nrhs[j]; ++rr, ++s) {
            const double2* src = (const double2*)bsrc[j] + (size_t)rr * n;
            if (host) {
                r = ovl_priv::ensure_base(c);
                if (r) return bfail(b, r, c->err);
                if (cudaMemcpyAsync(c->stage_in, src, vb, cudaMemcpyHostToDevice, st) != cudaSuccess)
                    return bfail(b, OVL_ECUDA, "source copy");
                src = c->stage_in;
            }
            ovl::launch_pack_spinor(src, b->b64[s], 0, c->g, st);
        }
    }
    // launch shapes: timed once per batch on its own data (short eager solves), unless OVL_NO_TUNE
    const int kind = tune_kind(b, flags);
    if (!b->pinned && b->tuned_kind != kind && !(flags & OVL_NO_TUNE)) {
        const std::string key = tune_key(b, kind);
        std::array<int, 3> v;
        if (tune_lookup(key, v)) {  // tuned before for this GPU, batch shape and precision
            b->shape = v[0], b->regen_minb = v[1], b->regen_pair = v[2];
            b->tuned = true;
            b->tuned_kind = kind;
            b->tune_cached = true;
            if (b->exec) cudaGraphExecDestroy(b->exec);
            b->exec = nullptr;
        } else {
            // both regenerations follow the same FP32 pass 1: its shape, and so its order of sums, is one choice
            std::array<int, 3> other;
            const bool shared = b->mode == 1 && tune_lookup(tune_key(b, kind == 1 ? 3 : 1), other);
            r = autotune(b, mu, kappa, flags, shared ? other[0] : -1, st);
            if (r) return r;
            b->tune_cached = false;
            tune_store(key, {b->shape, b->regen_minb, b->regen_pair});
        }
    }
    // the solve, as a graph captured once per (k, flags, mu, kappa); per-phase events need eager launches
    if (flags & OVL_PROFILE) {
        flags |= OVL_NO_GRAPH;
        for (cudaEvent_t& e : b->ev)
            if (!e && cudaEventCreate(&e) != cudaSuccess) return bfail(b, OVL_ECUDA, "profile events");
    }
    const int gflags = flags & (OVL_MIXED | OVL_NO_GRAPH | OVL_TWO_PASS | OVL_PASS2_F64 | OVL_STEPWISE);
    if (flags & OVL_NO_GRAPH) {
        r = enqueue_batch(b, k, mu, kappa, flags, st);
        if (r) return r;
    } else {
        std::vector<int> msig;
        for (const ovl_ctx* c : b->ctx) msig.push_back(c->m);
        if (!b->exec || b->g_k != k || b->g_flags != gflags || b->g_mu != mu || b->g_kappa != kappa ||
            b->g_m != msig) {
            if (b->exec) cudaGraphExecDestroy(b->exec);
            b->exec = nullptr;
            if (!b->cap_st && cudaStreamCreateWithFlags(&b->cap_st, cudaStreamNonBlocking) != cudaSuccess)
                return bfail(b, OVL_ECUDA, "capture stream");
            cudaGraph_t gr = nullptr;
            if (cudaStreamBeginCapture(b->cap_st, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
                return bfail(b, OVL_ECUDA, "begin capture");
            r = enqueue_batch(b, k, mu, kappa, flags, b->cap_st);
            cudaError_t e = cudaStreamEndCapture(b->cap_st, &gr);
            if (r) {
                if (gr) cudaGraphDestroy(gr);
                return r;
            }
            if (e != cudaSuccess) return bfail(b, OVL_ECUDA, std::string("end capture: ") + cudaGetErrorString(e));
            e = cudaGraphInstantiate(&b->exec, gr, 0);
            cudaGraphDestroy(gr);
            if (e != cudaSuccess) {
                b->exec = nullptr;
                return bfail(b, OVL_ECUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
            }
            b->g_k = k, b->g_flags = gflags, b->g_mu = mu, b->g_kappa = kappa;
            b->g_m = msig;
        }
        if (cudaGraphLaunch(b->exec, st) != cudaSuccess) return bfail(b, OVL_ECUDA, "graph launch");
    }
    // unpack: out = y, or D_ov b = b + gamma5 y with OVL_OVERLAP
    s = 0;
    for (size_t j = 0; j < b->ctx.size(); ++j) {
        ovl_ctx* c = b->ctx[j];
        const size_t n = c->n, vb = n * sizeof(double2);
        for (int rr = 0; rr < b->nrhs[j]; ++rr, ++s) {
            const double2* src = (const double2*)bsrc[j] + (size_t)rr * n;
            double2* dst = (double2*)out[j] + (size_t)rr * n;
            const bool ov = (flags & OVL_OVERLAP) != 0;
            if (host) {
                if (ov && cudaMemcpyAsync(c->stage_in, src, vb, cudaMemcpyHostToDevice, st) != cudaSuccess)
                    return bfail(b, OVL_ECUDA, "source copy");
                ovl::launch_unpack_spinor(b->hseq[s].y, 0, c->stage_out, ov ? c->stage_in : nullptr, ov ? 1 : 0, c->g,
                                          st);
                if (cudaMemcpyAsync(dst, c->stage_out, vb, cudaMemcpyDeviceToHost, st) != cudaSuccess)
                    return bfail(b, OVL_ECUDA, "result copy");
            } else {
                ovl::launch_unpack_spinor(b->hseq[s].y, 0, dst, ov ? src : nullptr, ov ? 1 : 0, c->g, st);
            }
        }
    }
    std::vector<ovl::KState> ks(b->nseq);
    if (cudaMemcpyAsync(ks.data(), b->ks, b->nseq * sizeof(ovl::KState), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return bfail(b, OVL_ECUDA, std::string("batch solve: ") + cudaGetErrorString(cudaGetLastError()));
    if (flags & OVL_PROFILE) {
        for (int j = 0; j < 3; ++j) {
            float ms = 0.f;
            cudaEventElapsedTime(&ms, b->ev[j], b->ev[j + 1]);
            b->prof_ms[j] += ms;
        }
        b->prof_n += 1;
    }
    int worst = OVL_OK;
    for (int q = 0; q < b->nseq; ++q) {
        if (info) {
            info[q].k_used = ks[q].kused;
            info[q].breakdown_step = ks[q].bdstep;
            info[q].inner_iters = ks[q].inner_iters;
            info[q].inner_method = ks[q].inner_method;
            info[q].bperp_norm = ks[q].nR;
            info[q].inner_err = ks[q].inner_err;
        }
        int code = OVL_OK;
        if (ks[q].timeout) code = OVL_ETIMEOUT;
        else if (ks[q].status) code = ks[q].status;
        else if (ks[q].bdstep >= 0) code = OVL_EBREAKDOWN;
        if (code && !worst) {
            worst = code;
            b->err = "sequence " + std::to_string(q) + " failed";
        }
    }
    return worst;
}

int ovl_batch_profile(ovl_batch* b, double* ms3, int* nsolves, int reset) {
    if (!b) return OVL_EINVAL;
    if (ms3)
        for (int j = 0; j < 3; ++j) ms3[j] = b->prof_ms[j];
    if (nsolves) *nsolves = b->prof_n;
    if (reset) {
        for (int j = 0; j < 3; ++j) b->prof_ms[j] = 0.0;
        b->prof_n = 0;
    }
    return OVL_OK;
}

int ovl_sign_krylov_batched(ovl_ctx* const* ctxs, int nctx, const int* nrhs, int k, double mu, double kappa,
                            const void* const* b, void* const* out, int flags, ovl_info* info) {
    ovl_batch* bt = nullptr;
    int r = ovl_batch_create(&bt, ctxs, nctx, nrhs);
    if (r) return r;
    r = ovl_batch_solve(bt, k, mu, kappa, b, out, flags | OVL_NO_GRAPH, info);
    if (r && ctxs[0]) ctxs[0]->err = bt->err;
    ovl_batch_destroy(bt);
    return r;
}

}  // extern "C"
