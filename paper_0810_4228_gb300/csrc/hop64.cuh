// The FP64 Wilson hop with a site shared by lanes (one hop, or one spin row of a hop, per lane): used by the
// FP64 stencil and the cooperative FP64 Krylov kernels.  A warp issues one FP64 instruction per 64 cycles
// and an SM one per 19 (measured), so lanes are filled and nothing that an integer instruction can do
// (sign changes) is left to the FP64 pipe.
#pragma once

#include "stencil_impl.cuh"

namespace ovl {

// chunk stride of a warp's half spinors: four groups (sites, or sites x inputs) of eight hops at a stride of
// nine slots, plus one, so that the epilogue's lanes fall into different banks
constexpr int HP_ST = 4 * 9 + 1;

// x with its sign bit flipped by mask (0 or 0x80000000): an integer operation (FP64 negation of a value
// that is not an operand of arithmetic runs on the FP64 pipe)
__device__ __forceinline__ double flip(double x, unsigned mask) {
    return __hiloint2double(__double2hiint(x) ^ (int)mask, __double2loint(x));
}
constexpr unsigned SIGN = 0x80000000u;

// Hop h (direction h & 3, forward for h < 4) of one site from x: U (or U^dag) times the projected half
// spinor, without the hop coefficient; both spin rows (RS = 1: o[0..2] row 0, o[3..5] row 1) or row `row`
// (RS = 2: o[0..2]).  xb: component 0 of the neighbour's spinor, components xs apart; ub: element 0 of the
// link (of the site itself, or of the neighbour for the backward hop), elements V apart; edge: the hop takes
// the phase -1.  CG: L2-coherent vector loads (vectors that other blocks of the kernel write).
template <int RS, bool CG>
__device__ __forceinline__ void hop_lane(int h, int row, const double2* xb, size_t xs, const double2* __restrict__ ub,
                                         size_t V, bool edge, cx<double> (&o)[6 / RS]) {
    const int nu = h & 3;
    const bool fwd = h < 4;
    const bool im = (nu & 1) == 0;
    cx<double> hh[2 / RS][3];
#pragma unroll
    for (int r = 0; r < 2 / RS; ++r) {
        const int rw = RS == 2 ? row : r;
        // row 0 takes spins 0 and 2 (nu >= 2) or 3, row 1 spins 1 and 3 or 2
        const double2* pb = xb + (size_t)(3 * rw) * xs;
        const double2* qb = xb + (size_t)((nu >= 2) == (rw == 0) ? 6 : 9) * xs;
        const bool neg = rw == 0 ? ((nu == 3) ? !fwd : fwd) : ((nu == 0) ? fwd : !fwd);
        const double s = neg ? -1.0 : 1.0, sr = neg != im ? -1.0 : 1.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double2 p = CG ? __ldcg(pb + a * xs) : __ldg(pb + a * xs);
            const double2 q = CG ? __ldcg(qb + a * xs) : __ldg(qb + a * xs);
            hh[r][a] = mk(fma(sr, im ? q.y : q.x, p.x), fma(s, im ? q.x : q.y, p.y));
        }
    }
    const size_t srow = fwd ? 3 * V : V, scol = fwd ? V : 3 * V;
    const unsigned pm = edge ? SIGN : 0u, cm = fwd ? pm : pm ^ SIGN;  // antiperiodic phase, conjugate
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double2 v = __ldg(ub + a * srow + k * scol);
            const cx<double> u = mk(flip(v.x, pm), flip(v.y, cm));
#pragma unroll
            for (int r = 0; r < 2 / RS; ++r) {
                if (k == 0) o[3 * r + a] = u * hh[r][0];
                else cfma(o[3 * r + a], u, hh[r][k]);
            }
        }
    }
}

// What the lane of (spin sp, part: 0 real, 1 imaginary) takes from hop w: slot of its half-spinor chunk
// (colour 0) and its coefficient in the sum of the hops: +-1 (exact), with e^{+-mu} on the temporal ones.
__device__ __forceinline__ void epilogue_lane(int sp, int part, double emu, double emum, int (&off)[8],
                                              double (&cw)[8]) {
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const int nu = w & 3;
        const bool fwd = w < 4, hi2 = nu >= 2, im = (nu & 1) == 0;
        int row = sp, pp = part;
        bool neg = false;
        if (sp >= 2) {
            row = hi2 ? sp - 2 : 3 - sp;
            const bool nA = !fwd, nB = (nu == 0 || nu == 3) ? !fwd : fwd;
            neg = (sp == 2 ? nA : nB) != (im && part == 0);
            if (im) pp = 1 - part;
        }
        off[w] = (row * 3 * HP_ST + w) * 2 + pp;
        cw[w] = flip(nu < 3 ? 1.0 : fwd ? emu : emum, neg ? SIGN : 0u);
    }
}
// The sum of the eight hops for one real number of the output; hd: the site's half spinors at the colour.
// kappa and the diagonal term are the caller's last fused multiply-add: the roundings of the sum then enter
// scaled by kappa (summing into the diagonal term gave 1.2 x the error of the one-thread-per-site form).
__device__ __forceinline__ double hop_sum(const double* hd, const int (&off)[8], const double (&cw)[8]) {
    double s = flip(hd[off[0]], (unsigned)__double2hiint(cw[0]) & SIGN);
#pragma unroll
    for (int w = 1; w < 8; ++w) s = fma(cw[w], hd[off[w]], s);
    return s;
}

}  // namespace ovl
