// Adjoint of y = A x, A = gamma5 D_w(mu; U) (Sec. 1, Eq. 1.2), for gradients of a
// real function l of y, in PyTorch's convention for complex tensors: the gradient
// of a complex z is g_z = dl/dRe z + i dl/dIm z (= 2 dl/dz*), so dl = Re <g_z, dz>
// with <a, b> = a^dag b.  With g = g_y:
//   grad_x        = A^dag g = gamma5 D_w(-mu) g                  (the stencil itself)
//   grad_U[x,nu]  = g_U
//                 = -kappa ( c+ ph sum_s g~_s (x) conj(psi(x+nu)_s)
//                          + c- ph sum_s psi(x)_s (x) conj(g^_s) ),
//        g~ = (1 + gamma_nu) gamma5 g(x),  g^ = (1 - gamma_nu) gamma5 g(x+nu),
//        (a (x) conj(b))_ij = a_i conj(b_j) in colour, c+- = e^{+-mu} for nu = 4
//        (1 otherwise), ph the antiperiodic phase of a hop across the time edge;
//   dl/dmu        = Re <g, (dA/dmu) x>,  dA/dmu = -kappa gamma5 (e^mu T_4^+ - e^-mu T_4^-).
// Every link receives the forward hop of its own site and the backward hop of
// the site it points to.  Canonical layouts in and out.
#include <cmath>

#include "ctx.h"
#include "force.cuh"

namespace ovl {
namespace {

// One link per thread, a warp per direction (32 consecutive sites of each of the four directions per block;
// the direction of a warp rotates with the block, so that the temporal links' extra work spreads over the
// SM quarters).  R = float: the spatial links in FP32 (OVL_F32); the temporal ones, whose forces also give
// d/dmu, stay FP64.  Bound by the FP64 pipe: 192 operations per link (force.cuh) and 54 for d/dmu; 24^4:
// 1490 -> 571 us against one thread per site with four-spin products and the temporal hops applied again.
template <class R, int NU>
__device__ __forceinline__ void link_grad(const double2* gx, const double2* gy, const double2* px, const double2* py,
                                          double2* o, double kappa, double ph) {
    cx<R> z[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) z[e] = mk(R(0), R(0));
    half_force<R, NU>(gx, gy, px, py, 1, z, z);
    const R f = -(R)kappa * (R)ph;
#pragma unroll
    for (int e = 0; e < 9; ++e) o[e] = make_double2((double)(f * z[e].r), (double)(f * z[e].i));
}

template <class R>
__global__ void __launch_bounds__(128, 4) k_dw_grad(const double2* __restrict__ U, const double2* __restrict__ x,
                                                 const double2* __restrict__ gr, double2* __restrict__ gU,
                                                 double kappa, double emu, double emum, Geom g, double* partials,
                                                 unsigned int* counter, double* gmu) {
    __shared__ double red[32];
    // (without the links' gradient: the temporal link of 128 sites per block)
    const int nu = gU ? ((threadIdx.x >> 5) + blockIdx.x) & 3 : 3;
    const int s = gU ? blockIdx.x * 32 + (threadIdx.x & 31) : blockIdx.x * 128 + threadIdx.x;
    double part[1] = {0.0};
    if (s < g.V) {
        int c[4], r = s;
        c[3] = r % g.L[3];
        r /= g.L[3];
        c[2] = r % g.L[2];
        r /= g.L[2];
        c[1] = r % g.L[1];
        c[0] = r / g.L[1];
        int y[4];
#pragma unroll
        for (int d = 0; d < 4; ++d) y[d] = d == nu ? (c[d] + 1 == g.L[d] ? 0 : c[d] + 1) : c[d];
        const size_t i = (size_t)s * 12, f = (size_t)canon_index(g, y) * 12;
        const double2 *gx = gr + i, *gy = gr + f, *px = x + i, *py = x + f;
        double2* o = gU + ((size_t)s * 4 + nu) * 9;
        switch (nu) {  // uniform per warp
            case 0: link_grad<R, 0>(gx, gy, px, py, o, kappa, 1.0); break;
            case 1: link_grad<R, 1>(gx, gy, px, py, o, kappa, 1.0); break;
            case 2: link_grad<R, 2>(gx, gy, px, py, o, kappa, 1.0); break;
            default: {
                cx<double> zf[9], zb[9];
#pragma unroll
                for (int e = 0; e < 9; ++e) zf[e] = zb[e] = mk(0.0, 0.0);
                half_force<double, 3>(gx, gy, px, py, 1, zf, zb);
                const double ph = c[3] == g.L[3] - 1 ? (double)g.bc_t : 1.0;
                const double af = -kappa * emu * ph, ab = -kappa * emum * ph;
                const double2* u = U + (size_t)27 * g.V + internal_index(g, c);
#pragma unroll
                for (int e = 0; e < 9; ++e) {
                    const cx<double> F = af * zf[e];
                    if (gU) o[e] = make_double2(fma(ab, zb[e].r, F.r), fma(ab, zb[e].i, F.i));
                    const double2 v = __ldg(u + (size_t)e * g.V);
                    part[0] = fma(v.x, fma(-ab, zb[e].r, F.r), part[0]);
                    part[0] = fma(v.y, fma(-ab, zb[e].i, F.i), part[0]);
                }
            }
        }
    }
    double out[1];
    if (grid_sum_last<1>(part, partials, counter, out, red))
        if (threadIdx.x == 0) *gmu = out[0];
}

}  // namespace
}  // namespace ovl

using namespace ovl_priv;

extern "C" int ovl_dw_grad(ovl_ctx* c, double mu, double kappa, const void* x, const void* g, void* grad_U,
                           double* grad_mu, int flags) {
    if (!c || !x || !g) return fail(c, OVL_EINVAL, "null argument");
    if (!c->have_gauge) return fail(c, OVL_ESTATE, "gauge field not set");
    if (flags & OVL_HOST) return fail(c, OVL_EINVAL, "device pointers only");
    if (flags & ~OVL_F32) return fail(c, OVL_EINVAL, "flags: 0 or OVL_F32");
    int r = ensure_solve(c, std::max(c->kcap, 1));
    if (r) return r;
    double* gmu = reinterpret_cast<double*>(c->h2);
    const int T = 128, per = grad_U ? 32 : T, B = (c->g.V + per - 1) / per;  // sites per block (k_dw_grad)
    if (flags & OVL_F32)
        ovl::k_dw_grad<float><<<B, T, 0, c->st>>>(c->U64, (const double2*)x, (const double2*)g, (double2*)grad_U,
                                                  kappa, exp(mu), exp(-mu), c->g, c->partials, c->counter, gmu);
    else
        ovl::k_dw_grad<double><<<B, T, 0, c->st>>>(c->U64, (const double2*)x, (const double2*)g, (double2*)grad_U,
                                                   kappa, exp(mu), exp(-mu), c->g, c->partials, c->counter, gmu);
    OVL_CUDA_TRY(c, cudaGetLastError());
    if (grad_mu) {
        OVL_CUDA_TRY(c, cudaMemcpyAsync(grad_mu, gmu, sizeof(double), cudaMemcpyDeviceToHost, c->st));
        OVL_CUDA_TRY(c, cudaStreamSynchronize(c->st));
    }
    return OVL_OK;
}
