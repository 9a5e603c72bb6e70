// The link force of y = A x in half spinors, shared by the derivative of A (grad.cu) and the FP64 derivative of
// the sign function (grad_krylov.cu; its mixed form has its own FP32 sum in full spinors).  With P = 1 + S gamma_nu (P^2 = 2 P, P^dag = P) and the reconstruction of P a
// from its upper two spins h_a,
//   sum_spins (P a)_i conj(b_j) = 1/2 sum_spins (P a)_i conj((P b)_j) = sum_{s = 0, 1} h_a,s,i conj(h_b,s,j),
// so the colour outer product of four spins takes two, 192 FP64 operations per link (48 projection sums, 144
// multiply-adds) instead of 520.  The mu derivative needs no hop of its own: Re <g, dA/dmu x> is
// Re sum_ij U_ij conj(F_ij) over the temporal links with the same F.
#pragma once

#include "stencil_impl.cuh"

namespace ovl {

template <class R> __device__ __forceinline__ cx<R> ld_as(const double2* p) {
    const double2 v = __ldg(p);
    return mk((R)v.x, (R)v.y);
}

// Colour a of spin ROW (0, 1) of (1 + S gamma_NU) psi; b: component 0 of psi, components st apart.
// (gamma5 psi in place of psi: S -> -S.)
template <class R, int NU, int S, int ROW>
__device__ __forceinline__ cx<R> proj_row(const double2* __restrict__ b, size_t st, int a) {
    constexpr int Q = NU < 2 ? 3 - ROW : 2 + ROW;  // the lower spin it takes
    constexpr int T = NU == 3 ? S : (NU == 0 || ROW == 0) ? -S : S;
    const cx<R> p = ld_as<R>(b + (3 * ROW + a) * st), q = ld_as<R>(b + (3 * Q + a) * st);
    if (NU == 0 || NU == 2) return T > 0 ? mk(p.r - q.i, p.i + q.r) : mk(p.r + q.i, p.i - q.r);
    return T > 0 ? p + q : p - q;
}

// zf_ij += sum_s h(g5 g(x))_i conj(h(psi(x + nu))_j) (1 + gamma_nu), zb_ij += sum_s h(psi(x))_i
// conj(h(g5 g(x + nu))_j) (1 - gamma_nu); zf and zb may be the same array.
template <class R, int NU, int ROW>
__device__ __forceinline__ void half_force_row(const double2* gx, const double2* gy, const double2* px,
                                               const double2* py, size_t st, cx<R> (&zf)[9], cx<R> (&zb)[9]) {
    cx<R> u[3], v[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = proj_row<R, NU, -1, ROW>(gx, st, a);
        v[a] = proj_row<R, NU, +1, ROW>(py, st, a);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) cfmac(zf[3 * i + j], v[j], u[i]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = proj_row<R, NU, -1, ROW>(px, st, a);
        v[a] = proj_row<R, NU, +1, ROW>(gy, st, a);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) cfmac(zb[3 * i + j], v[j], u[i]);
}
template <class R, int NU>
__device__ __forceinline__ void half_force(const double2* gx, const double2* gy, const double2* px, const double2* py,
                                           size_t st, cx<R> (&zf)[9], cx<R> (&zb)[9]) {
    half_force_row<R, NU, 0>(gx, gy, px, py, st, zf, zb);
    half_force_row<R, NU, 1>(gx, gy, px, py, st, zf, zb);
}

}  // namespace ovl
