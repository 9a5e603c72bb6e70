// Arnoldi (Sec. 2, Eq. 2.2-2.6; with LR deflation Sec. 3, Eq. 3.4) with the basis V_k stored as
// double-float pairs and the classical Gram-Schmidt (applied twice) evaluated in double-float
// arithmetic on the FP32 pipe.
//
// Step j of the Arnoldi relation A V_j = V_{j+1} H_j:  t = A v_j (FP64 stencil on the FP64 copy of
// v_j), h1 = V^dag t, t -= V h1, h2 = V^dag t, t -= V h2, H[0..j, j] = h1 + h2,
// H[j+1, j] = |t|, v_{j+1} = t / |t|.  The two passes over the stored basis per Gram-Schmidt sweep
// are the whole cost of the method at large k (Sec. 5); with FP64 arithmetic they run at the FP64
// issue rate, which on this GPU is far below what HBM delivers for 16 bytes per complex element.
// Double-float values (hi + lo, about 48 significant bits) take the same 16 bytes per complex
// element and their products and sums run on the FP32 pipe, so the sweeps become bandwidth
// bound.  The coefficients h, H and the inner sign stay FP64; every product enters its sum through
// the exact FMA split (dfacc), and every sum of per-lane, per-warp and per-block partials is
// deterministic (fixed order).
#include <algorithm>

#include "ovl_kernels.h"
#include "df32.cuh"

namespace ovl {

static constexpr int AD_T = 256;    // threads per block
static constexpr int AD_W = AD_T / 32;
static constexpr int AD_CH = 1024;  // elements of x per block in the many-vector dot

// Storage of one complex number here: {re.hi, im.hi, re.lo, im.lo}, so that the leading and the trailing
// parts are the operand pairs of the packed FP32x2 arithmetic (df32.cuh) as loaded.
__device__ __forceinline__ float4 to_f4(cx<df> z) { return make_float4(z.r.hi, z.i.hi, z.r.lo, z.i.lo); }
__device__ __forceinline__ cx<df> from_f4(float4 v) { return mk(df(v.x, v.z), df(v.y, v.w)); }

// Complex sums of products in packed form: A collects (a.r v.r, a.i v.i), B (a.r v.i, a.i v.r); the two
// halves of each are combined once at the end, so a term is 24 packed instructions and four moves (the
// swapped v) instead of 48 scalar ones.
struct PAcc {
    dfacc2 A, B;
};
__device__ __forceinline__ void pacc_zero(PAcc& p) {
    p.A.s = p.A.e = p.B.s = p.B.e = make_float2(0.f, 0.f);
}
__device__ __forceinline__ void pacc_add(PAcc& p, const float4& a, const float4& v) {
    const float2 ah = make_float2(a.x, a.y), al = make_float2(a.z, a.w);
    dfacc2_add(p.A, ah, al, make_float2(v.x, v.y), make_float2(v.z, v.w));
    dfacc2_add(p.B, ah, al, make_float2(v.y, v.x), make_float2(v.w, v.z));
}
// sum a v
__device__ __forceinline__ cx<df> pacc_product(const PAcc& p) {
    return mk(df(p.A.s.x, p.A.e.x) - df(p.A.s.y, p.A.e.y), df(p.B.s.x, p.B.e.x) + df(p.B.s.y, p.B.e.y));
}
// sum conj(v) a
__device__ __forceinline__ cx<df> pacc_dot(const PAcc& p) {
    return mk(df(p.A.s.x, p.A.e.x) + df(p.A.s.y, p.A.e.y), df(p.B.s.y, p.B.e.y) - df(p.B.s.x, p.B.e.x));
}

// sum over the 32 lanes of a warp (butterfly; every lane ends with the same value)
__device__ __forceinline__ df warp_sum_df(df a) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const df b(__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o));
        a = a + b;
    }
    return a;
}

// ------------------------------------------------------------------ helpers --
// xdf = x (FP64 -> double-float split), n complex values
__global__ void k_adf_todf(const double2* __restrict__ x, float4* __restrict__ xdf, const KState* ks, size_t n) {
    if (ks->done || ks->status) return;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        xdf[e] = to_f4(d2df(x[e]));
}

// v_1 = x / |x| (|x| = nR from the deflation split): the double-float split into V_0 and its
// exact FP64 value (hi + lo fits a double) into x64, the stencil's input of step 0
__global__ void k_adf_start(const double2* __restrict__ x, float4* __restrict__ v, double2* __restrict__ x64,
                            const KState* ks, size_t n) {
    if (ks->status || ks->nR == 0.0) return;
    const double s = 1.0 / ks->nR;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const double2 a = x[e];
        const cx<df> z = d2df(make_double2(a.x * s, a.y * s));
        v[e] = to_f4(z);
        x64[e] = df2d(z);
    }
}

// ---------------------------------------------------------- many-vector dot --
// The update sweep streams the basis from HBM with one 16-byte load per lane and a chain of
// dependent double-float operations behind it, so a warp has about one load in flight; L2
// prefetches a fixed distance ahead (no registers held) keep more bytes in flight per SM.
static constexpr int AD_PFV = 4;   // update: vectors (of this warp) ahead
__device__ __forceinline__ void prefetch_l2(const float4* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
// 16-byte asynchronous global -> shared copies (completion waited for per thread with
// cp.async.wait_group, a hardware wait)
__device__ __forceinline__ void cp_async16(float4* smem, const float4* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
// Vectors of the basis that two consecutive sweeps cannot both find in L2 are read as evict-first, so that
// the last ones (AD_KEEP bytes of 129 MB) stay there from sweep to sweep: k = 450 on 8^4 (a basis of up to
// 354 MB) 54.2 -> 52.1 ms.  A shorter basis has none of them.
static constexpr size_t AD_KEEP = (size_t)88 << 20;
__device__ __forceinline__ unsigned long long evict_first_policy() {
    unsigned long long p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void cp_async16_hint(float4* smem, const float4* gmem, unsigned long long pol) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(s), "l"(gmem), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ float4 ldg_hint(const float4* p, unsigned long long pol) {
    float4 v;
    asm("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p), "l"(pol));
    return v;
}
static int adf_cold(int nvec, size_t n) { return (int)std::max<long long>(0, nvec - (long long)(AD_KEEP / (n * sizeof(float4)))); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// stage 1, grid (chunks, vector groups): block (c, g) stages elements [c*AD_CH, (c+1)*AD_CH) of
// x in shared memory; warp w forms the partial dots V_l^dag x over that chunk for
// l = g*vpb + w, g*vpb + w + AD_W, ... < min(nvec, (g+1)*vpb).  The warp streams its
// (vector, tile of AD_SUB elements) pieces through two shared-memory tiles: the copy of the next
// tile is in flight while the current one is summed, so every warp keeps 4 KB of the basis in
// flight instead of one 16-byte load per lane.
static constexpr int AD_SUB = 256;
static size_t adf_dot_smem() { return sizeof(float4) * ((size_t)AD_CH + (size_t)AD_W * 2 * AD_SUB); }

__global__ void __launch_bounds__(AD_T) k_adf_dot(const float4* __restrict__ V, size_t ld, int nvec, int vpb,
                                                  const float4* __restrict__ x, double2* __restrict__ part,
                                                  size_t n, const KState* ks) {
    extern __shared__ float4 adf_sm[];
    float4* xs = adf_sm;
    if (ks->done || ks->status) return;
    const size_t base = (size_t)blockIdx.x * AD_CH;
    const int lim = (int)(n - base < (size_t)AD_CH ? n - base : (size_t)AD_CH);
    for (int q = threadIdx.x; q < lim; q += AD_T) xs[q] = x[base + q];
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4* wb = adf_sm + AD_CH + (size_t)wid * 2 * AD_SUB;
    const int l0 = blockIdx.y * vpb + wid;
    const int l1 = min(nvec, blockIdx.y * vpb + vpb);
    const int nv = l0 < l1 ? (l1 - l0 + AD_W - 1) / AD_W : 0;
    const int ntile = (lim + AD_SUB - 1) / AD_SUB;
    const int total = nv * ntile;
    // each lane copies (and later reads) the elements lane, lane + 32, ... of a tile
    auto issue = [&](int it) {
        const int a = it / ntile, si = it - a * ntile;
        const float4* src = V + (size_t)(l0 + a * AD_W) * ld + base + (size_t)si * AD_SUB;
        float4* dst = wb + (it & 1) * AD_SUB;
        const int cnt = min(AD_SUB, lim - si * AD_SUB);
        for (int u = lane; u < cnt; u += 32) cp_async16(dst + u, src + u);
        cp_async_commit();
    };
    if (total > 0) issue(0);
    PAcc acc;
    pacc_zero(acc);
    for (int it = 0; it < total; ++it) {
        if (it + 1 < total) {
            issue(it + 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncwarp();
        const int a = it / ntile, si = it - a * ntile;
        const float4* cur = wb + (it & 1) * AD_SUB;
        const float4* xt = xs + si * AD_SUB;
        const int cnt = min(AD_SUB, lim - si * AD_SUB);
        if (si == 0) pacc_zero(acc);
#pragma unroll 4
        for (int u = lane; u < cnt; u += 32) pacc_add(acc, xt[u], cur[u]);
        if (si == ntile - 1) {
            const cx<df> d = pacc_dot(acc);
            const df sr = warp_sum_df(d.r), si2 = warp_sum_df(d.i);
            if (lane == 0)
                part[(size_t)(l0 + a * AD_W) * gridDim.x + blockIdx.x] = make_double2(sr.to_double(), si2.to_double());
        }
        __syncwarp();  // this tile's buffer receives the copy issued two iterations on
    }
}

// stage 2: one warp per vector sums its block partials in FP64 (fixed order); h in FP64 and as a
// double-float split for the update kernels
__global__ void k_adf_dot_reduce(const double2* __restrict__ part, int nblk, int nvec, double2* __restrict__ h,
                                 float4* __restrict__ hdf, const KState* ks) {
    if (ks->done || ks->status) return;
    const int lane = threadIdx.x & 31;
    const int l = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (l >= nvec) return;
    double re = 0.0, im = 0.0;
    for (int b = lane; b < nblk; b += 32) {
        const double2 v = part[(size_t)l * nblk + b];
        re += v.x;
        im += v.y;
    }
    re = warp_sum(re);
    im = warp_sum(im);
    if (lane == 0) {
        h[l] = make_double2(re, im);
        hdf[l] = to_f4(d2df(make_double2(re, im)));
    }
}

// ------------------------------------------------------- many-vector update --
// Block = 32 consecutive elements (lane) x AD_W warps; warp w sums c_l V_l[e] over l = w, w + AD_W,
// ... < nvec, the warps' sums are added in shared memory in warp order.
__device__ __forceinline__ void adf_lincomb(const float4* __restrict__ V, size_t ld, int nvec,
                                            const float4* __restrict__ c, size_t e, bool in, int wid, int lane,
                                            float4 (&red)[AD_W][32], cx<df>& sum) {
    PAcc acc;
    pacc_zero(acc);
    if (in) {
#pragma unroll 4
        for (int l = wid; l < nvec; l += AD_W) {
            if ((lane & 7) == 0 && l + AD_PFV * AD_W < nvec)  // one lane per 128-byte line
                prefetch_l2(V + (size_t)(l + AD_PFV * AD_W) * ld + e);
            pacc_add(acc, __ldg(c + l), __ldg(V + (size_t)l * ld + e));
        }
    }
    red[wid][lane] = to_f4(pacc_product(acc));
    __syncthreads();
    if (wid == 0) {
        sum = from_f4(red[0][lane]);
#pragma unroll
        for (int w = 1; w < AD_W; ++w) sum = sum + from_f4(red[w][lane]);
    }
}

struct ArnoldiFinDf {
    double2* H;
    int ldH;
    const double2* h1;
    const double2* h2;
    int j;
    int jlast;
    double bdtol;  // lucky breakdown when H[j+1, j] <= bdtol * (largest column norm of H so far)
};

// x -= sum_l h_l V_l (x double-float, in place).  fin = 1 (second pass of step j): also |x|^2 over
// the grid, and the last block writes H[0..j, j] = h1 + h2, H[j+1, j] = |x|, kused = j + 1 and
// marks the solve done on a lucky breakdown or at j = jlast.
__global__ void __launch_bounds__(AD_T) k_adf_update(const float4* __restrict__ V, size_t ld, int nvec,
                                                     const float4* __restrict__ hdf, float4* __restrict__ x,
                                                     size_t n, KState* ks, int fin, ArnoldiFinDf af,
                                                     double* partials, unsigned int* counter) {
    __shared__ float4 red[AD_W][32];
    __shared__ double rsm[32];
    if (ks->done || ks->status) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t ntile = (n + 31) / 32;
    double part[1] = {0.0};
    for (size_t tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const size_t e = tile * 32 + lane;
        const bool in = e < n;
        cx<df> s;
        adf_lincomb(V, ld, nvec, hdf, e, in, wid, lane, red, s);
        if (wid == 0 && in) {
            const cx<df> xv = from_f4(x[e]);
            const cx<df> z = mk(xv.r - s.r, xv.i - s.i);
            x[e] = to_f4(z);
            const double2 zd = df2d(z);
            part[0] += zd.x * zd.x + zd.y * zd.y;
        }
        __syncthreads();  // red is reused by the next tile
    }
    if (!fin) return;
    double out[1];
    if (grid_sum_last<1>(part, partials, counter, out, rsm)) {
        const int j = af.j;
        double hh = 0.0;
        for (int r = threadIdx.x; r <= j; r += blockDim.x) {
            const double2 a = af.h1[r], b = af.h2[r];
            const double2 v = make_double2(a.x + b.x, a.y + b.y);
            af.H[r + (size_t)j * af.ldH] = v;
            hh += v.x * v.x + v.y * v.y;
        }
        double hv[1] = {hh};
        block_sum<1>(hv, rsm);
        if (threadIdx.x == 0) {
            const double hn = sqrt(out[0]);
            af.H[(j + 1) + (size_t)j * af.ldH] = make_double2(hn, 0.0);
            const double colnorm = sqrt(hv[0] + out[0]);
            if (colnorm > ks->anorm) ks->anorm = colnorm;
            ks->kused = j + 1;
            ks->red[0] = make_double2(hn, 0.0);
            if (hn <= af.bdtol * fmax(ks->anorm, 1e-300) || j == af.jlast) ks->done = 1;
        }
    }
}

// v_{j+1} = t / |t| in place (double-float), and its exact FP64 value into x64 (the next step's
// stencil input); skipped after the last step or a lucky breakdown
__global__ void k_adf_normalize(float4* __restrict__ t, double2* __restrict__ x64, const KState* ks, size_t n) {
    if (ks->done || ks->status) return;
    const df inv(1.0 / ks->red[0].x);
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const cx<df> z = from_f4(t[e]);
        const cx<df> v = mk(z.r * inv, z.i * inv);
        t[e] = to_f4(v);
        x64[e] = df2d(v);
    }
}

// c_l as double-float splits for l < kused
__global__ void k_adf_coef(const double2* __restrict__ c, float4* __restrict__ cdf, const KState* ks) {
    if (ks->status) return;
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < ks->kused; l += gridDim.x * blockDim.x)
        cdf[l] = to_f4(d2df(c[l]));
}

// y += sum_{l < kused} c_l V_l (Eq. 2.6), y FP64
__global__ void __launch_bounds__(AD_T) k_adf_combine(const float4* __restrict__ V, size_t ld,
                                                      const float4* __restrict__ cdf, const KState* ks,
                                                      double2* __restrict__ y, size_t n) {
    __shared__ float4 red[AD_W][32];
    if (ks->status) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t e = (size_t)blockIdx.x * 32 + lane;
    const bool in = e < n;
    cx<df> s;
    adf_lincomb(V, ld, ks->kused, cdf, e, in, wid, lane, red, s);
    if (wid == 0 && in) {
        const double2 a = y[e], d = df2d(s);
        y[e] = make_double2(a.x + d.x, a.y + d.y);
    }
}

// ================================================== low-synch Arnoldi: delayed CGS2 ==
// Classical Gram-Schmidt applied twice with the second pass delayed by one step (the "DCGS2" of the
// low-synchronisation Gram-Schmidt literature: Swirydowicz, Langou, Ananthan, Yang and Thomas,
// Numer. Linear Algebra Appl. 28 (2021); Bielich, Langou, Thomas, Swirydowicz, Yamazaki and Boman,
// Parallel Comput. 112 (2022)), on the double-float basis.  At step j the slots V_0..V_{j-1} hold
// final orthonormal vectors and slot j holds u_j, A v_{j-1} projected once and neither
// re-orthogonalised nor normalised; the stencil has produced w = A u_j (FP64) from its FP64 value.
//  (1) one sweep over V_0..V_j:  c = V_{<j}^dag u_j, rho^2 = u_j^dag u_j, d = V_{<j}^dag w,
//      e = u_j^dag w                                           (k_adf_dot2, k_adf_dot2_reduce)
//  (2) nu^2 = rho^2 - |c|^2 (V_{<j} orthonormal); column j-1 of H becomes final,
//      H[<j, j-1] += c, H[j, j-1] = nu; v_j = (u_j - V_{<j} c) / nu             (k_adf_dcgs)
//  (3) one sweep over V_0..V_{j-1}:  v_j, and u_{j+1} = A v_j - V_{<=j} h = w / nu - V_{<j} d / nu
//      - r v_j with r = (e - c^dag d) / nu^2; the tentative column j of H is
//      h = (d / nu - g, r - c_{j-1}), g = H[<=j, <j] c / nu                      (k_adf_update2)
// because A v_j = (w - A V_{<j} c) / nu = (w - V_{<=j} H[<=j, <j] c) / nu by the Arnoldi relation
// of the final columns: the projection coefficients of A v_j come from the sums of (1) without
// another pass, and the basis is read twice per step instead of four times.  After the last step
// one more dot sweep re-orthogonalises u_k and finishes column k-1.  In exact arithmetic this is
// the Arnoldi process of Sec. 2 (Eq. 2.2-2.3).

// Bound by the FP32 pipe (24 packed operations per term, 58 % of its rate) beside 16 bytes of basis per term.
// All sweeps of k = 450 on 8^4: 29 ms in scalar arithmetic, 24.4 ms packed.
// Chunks of 512 elements and staging tiles of 128: 48 KB per block, four blocks (32 warps) per SM, and tasks
// (one vector over one chunk) small enough that the last round of warps costs little.
static constexpr int D2_CH = 512, D2_SUB = 128;
static size_t adf_dot2_smem() { return sizeof(float4) * (2 * (size_t)D2_CH + (size_t)AD_W * 2 * D2_SUB); }

// Warp sums of the four real numbers of two complex ones, transposed (6 double-float additions instead of
// 20): lanes 0, 8, 16, 24 end with a.r, a.i, b.r, b.i.
__device__ __forceinline__ df warp_sum4_df(const cx<df>& a, const cx<df>& b) {
    const int lane = threadIdx.x & 31;
    auto xchg = [](df x, int o) {
        return df(__shfl_xor_sync(0xffffffffu, x.hi, o), __shfl_xor_sync(0xffffffffu, x.lo, o));
    };
    const bool u16 = lane & 16, u8 = lane & 8;
    const df p = (u16 ? b.r : a.r) + xchg(u16 ? a.r : b.r, 16);
    const df q = (u16 ? b.i : a.i) + xchg(u16 ? a.i : b.i, 16);
    df r = (u8 ? q : p) + xchg(u8 ? p : q, 8);
    r = r + xchg(r, 4);
    r = r + xchg(r, 2);
    return r + xchg(r, 1);
}

// stage 1 of the two-vector dot, grid (chunks, vector groups): V_l^dag x1 and V_l^dag x2 for every
// l < nvec over the block's chunk; x1 is a double-float vector, x2 an FP64 one (split on staging).
// Partials: part[(2 l + q) * gridDim.x + chunk], q = 0 for x1, 1 for x2.
__global__ void __launch_bounds__(AD_T, 4) k_adf_dot2(const float4* __restrict__ V, size_t ld, int nvec, int vpb, int cold,
                                                   const float4* __restrict__ x1, const double2* __restrict__ x2,
                                                   double2* __restrict__ part, size_t n, const KState* ks) {
    extern __shared__ float4 adf_sm[];
    float4* xs1 = adf_sm;
    float4* xs2 = adf_sm + D2_CH;
    if (ks->done || ks->status) return;
    const size_t base = (size_t)blockIdx.x * D2_CH;
    const int lim = (int)(n - base < (size_t)D2_CH ? n - base : (size_t)D2_CH);
    for (int q = threadIdx.x; q < lim; q += AD_T) {
        xs1[q] = x1[base + q];
        xs2[q] = to_f4(d2df(x2[base + q]));
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4* wb = adf_sm + 2 * D2_CH + (size_t)wid * 2 * D2_SUB;
    const int l0 = blockIdx.y * vpb + wid;
    const int l1 = min(nvec, blockIdx.y * vpb + vpb);
    const int nv = l0 < l1 ? (l1 - l0 + AD_W - 1) / AD_W : 0;
    const int ntile = (lim + D2_SUB - 1) / D2_SUB;
    const int total = nv * ntile;
    const unsigned long long pol = evict_first_policy();
    auto issue = [&](int it) {
        const int a = it / ntile, si = it - a * ntile;
        const float4* src = V + (size_t)(l0 + a * AD_W) * ld + base + (size_t)si * D2_SUB;
        float4* dst = wb + (it & 1) * D2_SUB;
        const int cnt = min(D2_SUB, lim - si * D2_SUB);
        if (l0 + a * AD_W < cold)
            for (int u = lane; u < cnt; u += 32) cp_async16_hint(dst + u, src + u, pol);
        else
            for (int u = lane; u < cnt; u += 32) cp_async16(dst + u, src + u);
        cp_async_commit();
    };
    if (total > 0) issue(0);
    PAcc a1, a2;
    pacc_zero(a1);
    pacc_zero(a2);
    for (int it = 0; it < total; ++it) {
        if (it + 1 < total) {
            issue(it + 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncwarp();
        const int a = it / ntile, si = it - a * ntile;
        const float4* cur = wb + (it & 1) * D2_SUB;
        const int cnt = min(D2_SUB, lim - si * D2_SUB);
        if (si == 0) {
            pacc_zero(a1);
            pacc_zero(a2);
        }
#pragma unroll 4
        for (int u = lane; u < cnt; u += 32) {
            const float4 v = cur[u];
            pacc_add(a1, xs1[si * D2_SUB + u], v);
            pacc_add(a2, xs2[si * D2_SUB + u], v);
        }
        if (si == ntile - 1) {
            const cx<df> d1 = pacc_dot(a1), d2 = pacc_dot(a2);
            const df r = warp_sum4_df(d1, d2);
            if ((lane & 7) == 0) {
                const size_t l = (size_t)(l0 + a * AD_W);
                reinterpret_cast<double*>(part + (2 * l + (lane >> 4)) * gridDim.x + blockIdx.x)[(lane >> 3) & 1] =
                    r.to_double();
            }
        }
        __syncwarp();  // this tile's buffer receives the copy issued two iterations on
    }
}

// (2), one block of 256 threads.  h1 = (c, rho^2) and h2 = (d, e) of step j (h2 unused when fin).  Finishes
// column j-1 of H (j >= 1), decides a lucky breakdown (nu <= bdtol |H|) and for the update writes
// ks->red[1] = (1 / nu, nu), ks->red[2] = r.  fin = 1 after the
// last step (j = k): only column k-1 is finished and the solve is marked done.  fin = 2 at the end of a
// restart cycle: column k-1 is finished and ks->red[1] written for the next cycle's start vector
// (u_k - V c) / nu, and the solve goes on unless the Krylov space is invariant.
// FP64 instructions take 64 cycles of their warp each: the four sums are transposed over the warp (6
// additions instead of 20), nu comes from one reciprocal square root, and the column norm's own square root
// is taken by another warp.
static constexpr int DC_T = 256;
__device__ __forceinline__ void dcgs_block(double2* __restrict__ H, int ldH, const double2* h1, const double2* h2,
                                           KState* ks, int j, int fin, double bdtol) {
    __shared__ double red[DC_T / 32][4];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // |c|^2, c^dag d, |H[<j, j-1] + c|^2
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
    for (int l = threadIdx.x; l < j; l += DC_T) {
        const double2 c = __ldcg(h1 + l);
        a0 = fma(c.x, c.x, fma(c.y, c.y, a0));
        if (!fin) {
            const double2 d = __ldcg(h2 + l);
            a1 = fma(c.x, d.x, fma(c.y, d.y, a1));
            a2 = fma(c.x, d.y, fma(-c.y, d.x, a2));
        }
        double2* hp = H + l + (size_t)(j - 1) * ldH;
        double2 hv = *hp;
        hv.x += c.x;
        hv.y += c.y;
        *hp = hv;
        a3 = fma(hv.x, hv.x, fma(hv.y, hv.y, a3));
    }
    {
        const bool u16 = lane & 16, u8 = lane & 8;
        const double b0 = (u16 ? a2 : a0) + __shfl_xor_sync(0xffffffffu, u16 ? a0 : a2, 16);
        const double b1 = (u16 ? a3 : a1) + __shfl_xor_sync(0xffffffffu, u16 ? a1 : a3, 16);
        double r = (u8 ? b1 : b0) + __shfl_xor_sync(0xffffffffu, u8 ? b0 : b1, 8);
        r += __shfl_xor_sync(0xffffffffu, r, 4);
        r += __shfl_xor_sync(0xffffffffu, r, 2);
        r += __shfl_xor_sync(0xffffffffu, r, 1);
        if ((lane & 7) == 0) red[wid][lane >> 3] = r;  // lanes 0, 8, 16, 24: values 0, 1, 2, 3
    }
    __syncthreads();
    if (wid >= 2) return;
    double t = red[lane >> 2][lane & 3];
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    t += __shfl_xor_sync(0xffffffffu, t, 8);
    t += __shfl_xor_sync(0xffffffffu, t, 4);
    const double c2 = __shfl_sync(0xffffffffu, t, 0), er = __shfl_sync(0xffffffffu, t, 1);
    const double ei = __shfl_sync(0xffffffffu, t, 2), hn2 = __shfl_sync(0xffffffffu, t, 3);
    if (lane) return;
    const double rho2 = __ldcg(&h1[j].x), nu2 = rho2 - c2;
    if (wid == 1) {  // |H| so far, in the record of the next steps (warp 0 works with its square)
        if (j >= 1) {
            const double an = sqrt(hn2 + (nu2 > 0.0 ? nu2 : 0.0));
            if (an > ks->red[0].y) ks->red[0].y = an;
            ks->anorm = ks->red[0].y;
        }
        return;
    }
    const double inu = nu2 > 0.0 ? rsqrt(nu2) : 0.0, nu = nu2 > 0.0 ? nu2 * inu : 0.0;
    int stop = 0;
    if (j >= 1) {
        H[j + (size_t)(j - 1) * ldH] = make_double2(nu, 0.0);
        const double an2 = fmax(fmax(ks->red[0].x, hn2 + nu * nu), 1e-300);  // largest column so far, squared
        ks->red[0].x = an2;
        ks->kused = j;
        if (fin == 1 || nu * nu <= bdtol * bdtol * an2) stop = 1;  // last column, or K_j invariant
    } else if (!(nu > 0.0)) {
        stop = 1;  // zero start vector (cannot happen after the deflation split's check)
    }
    if (stop) {
        ks->done = 1;
        return;
    }
    ks->red[1] = make_double2(inu, nu);
    if (!fin) {  // r = (e - c^dag d) / nu^2
        const double2 e = __ldcg(h2 + j);
        const double i2 = inu * inu;
        ks->red[2] = make_double2((e.x - er) * i2, (e.y - ei) * i2);
    }
}

__global__ void __launch_bounds__(DC_T) k_adf_dcgs(double2* __restrict__ H, int ldH, const double2* __restrict__ h1,
                                                   const double2* __restrict__ h2, KState* ks, int j, int fin,
                                                   double bdtol) {
    if (ks->done || ks->status) return;
    dcgs_block(H, ldH, h1, h2, ks, j, fin, bdtol);
}

// stage 2 of the two-vector dot: one warp per (vector, operand) sums its chunk partials in FP64 (fixed
// order): h1[l] = V_l^dag x1, h2[l] = V_l^dag x2, and their double-float splits for the update; the last
// block to finish goes on with (2) (a launch of its own, a chain of FP64 instructions in one block, took 16 us of each step; in all
// 7.2 ms of k = 450 on 8^4, now 4.7 ms with the dot's second stage).
__global__ void __launch_bounds__(DC_T) k_adf_dot2_reduce(const double2* __restrict__ part, int nblk, int nvec,
                                                          double2* h1, double2* h2, float4* __restrict__ h1d,
                                                          float4* __restrict__ h2d, double2* __restrict__ H, int ldH,
                                                          KState* ks, double bdtol, unsigned int* counter) {
    __shared__ bool last;
    if (ks->done || ks->status) return;
    const int lane = threadIdx.x & 31;
    const int p = blockIdx.x * (DC_T / 32) + (threadIdx.x >> 5);
    if (p < 2 * nvec) {
        double re = 0.0, im = 0.0;
        for (int b = lane; b < nblk; b += 32) {
            const double2 v = part[(size_t)p * nblk + b];
            re += v.x;
            im += v.y;
        }
        // even lanes end with the real part's sum, odd lanes with the imaginary part's
        const bool odd = lane & 1;
        double r = (odd ? im : re) + __shfl_xor_sync(0xffffffffu, odd ? re : im, 1);
#pragma unroll
        for (int o = 2; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        const double ri = __shfl_sync(0xffffffffu, r, 1);
        if (lane == 0) {
            ((p & 1) ? h2 : h1)[p >> 1] = make_double2(r, ri);
            ((p & 1) ? h2d : h1d)[p >> 1] = to_f4(d2df(make_double2(r, ri)));
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x == 0) *counter = 0u;
    dcgs_block(H, ldH, h1, h2, ks, nvec - 1, 0, bdtol);
}

// (3): per element e, over the final vectors V_0..V_{j-1}: s1 = sum_l c_l V_l[e], s2 = sum_l d_l V_l[e];
// then v_j = (u_j - s1) / nu into slot j (in place of u_j) and u_{j+1} = (w - s2) / nu - r v_j into slot
// j + 1 and, as FP64, into x64 (the next stencil's input).  The first hb blocks write the tentative column j
// of H, a warp per row: H[i, j] = d_i / nu - g_i (i < j), r - c_{j-1} (i = j), g_i = sum_{l >= i-1} H[i, l] c_l / nu (upper
// Hessenberg rows of the final columns).
// Bound by the FP32 pipe (48 packed operations per term, both sums double-float) beside 16 bytes of basis per term.
// The 450 updates of k = 450 on 8^4: 30.1 ms with scalar sums, 24.0 ms so.  The solve takes 56.5 ms with two vectors per
// round at 32 warps per SM, 56.6 with four at 24 warps, 57.5 with two at 24, 58.7 and 59.2 with four and eight at 16.  (The
// c sum in FP32 from the leading parts, where |c| is small, takes 51.8: less than the basis's precision, not kept.)
static constexpr int UP_CH = 512;  // coefficients staged in shared memory at a time (a multiple of UP_NV x AD_W)
static constexpr int UP_NV = 2;   // vectors per warp and round
__global__ void __launch_bounds__(AD_T, 4) k_adf_update2(const float4* __restrict__ V, size_t ld, int j, int cold, int hb,
                                                         const float4* __restrict__ cdf, const float4* __restrict__ ddf,
                                                         float4* __restrict__ uj, float4* __restrict__ unext,
                                                         const double2* __restrict__ w, double2* __restrict__ x64,
                                                         double2* __restrict__ H, int ldH,
                                                         const double2* __restrict__ h1, const double2* __restrict__ h2,
                                                         size_t n, KState* ks) {
    __shared__ float4 red1[AD_W][32];
    __shared__ float4 red2[AD_W][32];
    __shared__ float4 csm[UP_CH], dsm[UP_CH];
    if (ks->done || ks->status) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double inu = ks->red[1].x;
    const double2 r = ks->red[2];
    if ((int)blockIdx.x < hb) {  // a warp per row of H
        const int i = blockIdx.x * AD_W + wid;
        if (i > j) return;
        double gr = 0.0, gi = 0.0;
        for (int l = max(i - 1, 0) + lane; l < j; l += 32) {
            const double2 hv = H[i + (size_t)l * ldH], c = h1[l];
            gr = fma(hv.x, c.x, fma(-hv.y, c.y, gr));
            gi = fma(hv.x, c.y, fma(hv.y, c.x, gi));
        }
        gr = warp_sum(gr) * inu;
        gi = warp_sum(gi) * inu;
        if (lane == 0) {
            double2 hv;
            if (i < j) {
                const double2 d = h2[i];
                hv = make_double2(d.x * inu - gr, d.y * inu - gi);
            } else {
                const double2 cl = j > 0 ? h1[j - 1] : make_double2(0.0, 0.0);
                hv = make_double2(r.x - cl.x, r.y - cl.y);
            }
            H[i + (size_t)j * ldH] = hv;
        }
        return;
    }
    const df dinu(inu);
    const cx<df> rr = d2df(r);
    const size_t ntile = (n + 31) / 32;
    const unsigned long long pol = evict_first_policy();
    for (size_t tile = blockIdx.x - hb; tile < ntile; tile += gridDim.x - hb) {
        const size_t e = tile * 32 + lane;
        const bool in = e < n;
        PAcc a1, a2;
        pacc_zero(a1);
        pacc_zero(a2);
        // UP_NV vectors of this warp per round, the next round's loads in flight meanwhile
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4* Ve = V + e;
        auto load = [&](int l, float4 (&v)[UP_NV]) {
#pragma unroll
            for (int q = 0; q < UP_NV; ++q) {
                const float4* p = Ve + (size_t)(l + q * AD_W) * ld;
                v[q] = !in || l + q * AD_W >= j ? zero : l < cold ? ldg_hint(p, pol) : __ldg(p);
            }
        };
        float4 v[UP_NV];
        load(wid, v);
        for (int l0 = 0; l0 < j; l0 += UP_CH) {
            if (l0 > 0 || tile + hb != blockIdx.x) __syncthreads();  // the last chunk has been read
            for (int l = threadIdx.x; l < UP_CH; l += AD_T) {
                const bool ok = l0 + l < j;
                csm[l] = ok ? __ldg(cdf + l0 + l) : zero;
                dsm[l] = ok ? __ldg(ddf + l0 + l) : zero;
            }
            __syncthreads();
            const int lim = min(UP_CH, j - l0);
            for (int l = wid; l < lim; l += UP_NV * AD_W) {
                float4 nx[UP_NV];
                load(l0 + l + UP_NV * AD_W, nx);
#pragma unroll
                for (int q = 0; q < UP_NV; ++q) {
                    pacc_add(a1, csm[l + q * AD_W], v[q]);
                    pacc_add(a2, dsm[l + q * AD_W], v[q]);
                    v[q] = nx[q];
                }
            }
        }
        red1[wid][lane] = to_f4(pacc_product(a1));
        red2[wid][lane] = to_f4(pacc_product(a2));
        __syncthreads();
        if (wid == 0 && in) {
            cx<df> s1 = from_f4(red1[0][lane]);
            cx<df> s2 = from_f4(red2[0][lane]);
#pragma unroll
            for (int q = 1; q < AD_W; ++q) {
                s1 = s1 + from_f4(red1[q][lane]);
                s2 = s2 + from_f4(red2[q][lane]);
            }
            const cx<df> u = from_f4(uj[e]);
            const cx<df> vj = mk((u.r - s1.r) * dinu, (u.i - s1.i) * dinu);
            const cx<df> ww = d2df(w[e]);
            const cx<df> rv = rr * vj;
            const cx<df> un = mk((ww.r - s2.r) * dinu - rv.r, (ww.i - s2.i) * dinu - rv.i);
            uj[e] = to_f4(vj);
            unext[e] = to_f4(un);
            x64[e] = df2d(un);
        }
        __syncthreads();  // red1, red2 are reused by the next tile
    }
}

// ======================================================== restarted Arnoldi ==
// Arnoldi restarted every m steps (Eiermann and Ernst, SIAM J. Numer. Anal. 44 (2006)): cycle c
// runs m delayed-CGS2 steps on the double-float basis slots 0..m from the start vector in slot 0,
// writing its Hessenberg block into the accumulated matrix at rows and columns c m ..; the block's
// subdiagonal entry H[m, m-1] is the coupling to the next cycle.  After the cycle the inner sign of
// the accumulated K x K matrix gives c_K = |b_perp| sgn(H_K) e_1, of which the rows of cycle c
// multiply its basis: y += V_c c_K[c m ..].  The next cycle starts from v_m = (u_m - V c) / nu.
// Cycle bookkeeping in the state record: red[4].x = K (columns finished so far), red[5] = (steps of
// this cycle, stopped); a lucky breakdown stops the process after that cycle's combination.
__global__ void k_rs_begin(KState* ks, int cyc) {
    if (ks->status) return;
    if (cyc == 0) {  // a source the deflation split left empty (done already) stops the process
        ks->red[4] = make_double2(0.0, 0.0);
        ks->red[5] = make_double2(0.0, ks->done ? 1.0 : 0.0);
    }
    ks->done = ks->red[5].y != 0.0 ? 1 : 0;
    ks->kused = 0;
}

// after the cycle's last Gram-Schmidt: K += steps of this cycle; kused = K for the inner sign
__global__ void k_rs_mid(KState* ks) {
    if (ks->status) return;
    const int local = ks->red[5].y != 0.0 ? 0 : ks->kused;
    const int K = (int)ks->red[4].x + local;
    ks->red[4] = make_double2((double)K, 0.0);
    ks->red[5].x = (double)local;
    ks->kused = K;
}

// double-float combination coefficients of this cycle: cdf[l] = c[off + l], l < steps
__global__ void k_rs_coef(const double2* __restrict__ c, float4* __restrict__ cdf, const KState* ks, int off) {
    if (ks->status) return;
    const int local = (int)ks->red[5].x;
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < local; l += gridDim.x * blockDim.x)
        cdf[l] = to_f4(d2df(c[off + l]));
}

// y += sum_{l < steps} cdf_l V_l (y FP64)
__global__ void __launch_bounds__(AD_T) k_rs_combine(const float4* __restrict__ V, size_t ld,
                                                     const float4* __restrict__ cdf, const KState* ks,
                                                     double2* __restrict__ y, size_t n) {
    __shared__ float4 red[AD_W][32];
    if (ks->status) return;
    const int local = (int)ks->red[5].x;
    if (local <= 0) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t e = (size_t)blockIdx.x * 32 + lane;
    const bool in = e < n;
    cx<df> s;
    adf_lincomb(V, ld, local, cdf, e, in, wid, lane, red, s);
    if (wid == 0 && in) {
        const double2 a = y[e], d = df2d(s);
        y[e] = make_double2(a.x + d.x, a.y + d.y);
    }
}

// the next cycle's start vector v_0 = (u_m - V_{<m} c) / nu into slot 0 (each element is read and
// written by its own block) and its FP64 value into x64; after the last cycle, a lucky breakdown
// or an earlier stop, the process is marked stopped and done instead
__global__ void __launch_bounds__(AD_T) k_rs_restart(float4* __restrict__ V, size_t ld, int m,
                                                     const float4* __restrict__ cdf, double2* __restrict__ x64,
                                                     KState* ks, size_t n, int last) {
    __shared__ float4 red[AD_W][32];
    if (ks->status) return;
    if (ks->done || ks->red[5].y != 0.0 || last) {  // the same decision in every block
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            ks->red[5].y = 1.0;
            ks->done = 1;
        }
        return;
    }
    const df inu(ks->red[1].x);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t ntile = (n + 31) / 32;
    for (size_t tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const size_t e = tile * 32 + lane;
        const bool in = e < n;
        cx<df> s;
        adf_lincomb(V, ld, m, cdf, e, in, wid, lane, red, s);
        if (wid == 0 && in) {
            const cx<df> u = from_f4(V[(size_t)m * ld + e]);
            const cx<df> v = mk((u.r - s.r) * inu, (u.i - s.i) * inu);
            V[e] = to_f4(v);
            x64[e] = df2d(v);
        }
        __syncthreads();  // red is reused by the next tile
    }
}

// ---------------------------------------------------------------- launchers --
// the update kernel's grid: one block per 32 elements up to AD_MAXB blocks (its norm partials,
// one double per block, must fit the solve's partials buffer of at least 2^16 doubles)
static constexpr unsigned AD_MAXB = 16384;
static unsigned adf_update_grid(size_t n) {
    const size_t t = (n + 31) / 32;
    return (unsigned)(t < AD_MAXB ? (t ? t : 1) : AD_MAXB);
}

static int adf_grid(size_t n) {
    size_t b = (n + 255) / 256;
    return (int)(b < 1024 ? (b ? b : 1) : 1024);
}

void launch_adf_todf(const double2* x, float4* xdf, const KState* ks, size_t n, cudaStream_t st) {
    k_adf_todf<<<adf_grid(n), 256, 0, st>>>(x, xdf, ks, n);
}

void launch_adf_start(const double2* x, float4* v, double2* x64, const KState* ks, size_t n, cudaStream_t st) {
    k_adf_start<<<adf_grid(n), 256, 0, st>>>(x, v, x64, ks, n);
}

int adf_dot_blocks(size_t n) { return (int)((n + AD_CH - 1) / AD_CH); }

void launch_adf_dot(const float4* V, size_t ld, int nvec, const float4* x, double2* h, float4* hdf,
                    double* partials, size_t n, int num_sms, const KState* ks, cudaStream_t st) {
    if (nvec <= 0) return;
    const int nchunk = adf_dot_blocks(n);
    // vectors per warp: about eight blocks per SM in total (four waves of the two that fit an SM with
    // their 80 KB of shared memory), at least one vector per warp
    const long long target = 8ll * (num_sms > 0 ? num_sms : 1);
    long long vpw = ((long long)nvec * nchunk + (long long)AD_W * target - 1) / ((long long)AD_W * target);
    if (vpw < 1) vpw = 1;
    const int vpb = (int)(vpw * AD_W);
    const int ngroup = (nvec + vpb - 1) / vpb;
    double2* part = reinterpret_cast<double2*>(partials);
    static unsigned long long attr_dev = 0;
    if (first_use_on_device(attr_dev))
        cudaFuncSetAttribute(k_adf_dot, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)adf_dot_smem());
    k_adf_dot<<<dim3(nchunk, ngroup), AD_T, adf_dot_smem(), st>>>(V, ld, nvec, vpb, x, part, n, ks);
    k_adf_dot_reduce<<<(nvec + 7) / 8, 256, 0, st>>>(part, nchunk, nvec, h, hdf, ks);
}

void launch_adf_update(const float4* V, size_t ld, int nvec, const float4* hdf, float4* x, size_t n, KState* ks,
                       double* partials, unsigned int* counter, cudaStream_t st) {
    if (nvec <= 0) return;
    ArnoldiFinDf af = {nullptr, 0, nullptr, nullptr, 0, 0, 0.0};
    k_adf_update<<<adf_update_grid(n), AD_T, 0, st>>>(V, ld, nvec, hdf, x, n, ks, 0, af, partials, counter);
}

void launch_adf_update_fin(const float4* V, size_t ld, int nvec, const float4* hdf, float4* x, double2* H, int ldH,
                           const double2* h1, const double2* h2, int j, int jlast, double* partials,
                           unsigned int* counter, KState* ks, size_t n, cudaStream_t st) {
    // double-float sweeps leave a residual of about 2^-46 |A v_j| where the Krylov space is
    // exhausted (FP64: 2^-53), so the breakdown test sits at 1e-11 instead of FP64's 1e-13
    ArnoldiFinDf af = {H, ldH, h1, h2, j, jlast, 1e-11};
    k_adf_update<<<adf_update_grid(n), AD_T, 0, st>>>(V, ld, nvec, hdf, x, n, ks, 1, af, partials, counter);
}

void launch_adf_normalize(float4* t, double2* x64, const KState* ks, size_t n, cudaStream_t st) {
    k_adf_normalize<<<adf_grid(n), 256, 0, st>>>(t, x64, ks, n);
}

// steps (1) and (2) of step nvec - 1
void launch_adf_dot2(const float4* V, size_t ld, int nvec, const float4* x1, const double2* x2, double2* h1,
                     double2* h2, float4* h1d, float4* h2d, double2* H, int ldH, double* partials,
                     unsigned int* counter, size_t n, int num_sms, KState* ks, cudaStream_t st) {
    if (nvec <= 0) return;
    const int nchunk = (int)((n + D2_CH - 1) / D2_CH);
    // vectors per warp: about 24 blocks per SM in all (six rounds of the four that fit an SM)
    const long long target = 24ll * (num_sms > 0 ? num_sms : 1);
    long long vpw = ((long long)nvec * nchunk + (long long)AD_W * target - 1) / ((long long)AD_W * target);
    if (vpw < 1) vpw = 1;
    const int vpb = (int)(vpw * AD_W);
    const int ngroup = (nvec + vpb - 1) / vpb;
    double2* part = reinterpret_cast<double2*>(partials);
    static unsigned long long attr_dev = 0;
    if (first_use_on_device(attr_dev))
        cudaFuncSetAttribute(k_adf_dot2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)adf_dot2_smem());
    k_adf_dot2<<<dim3(nchunk, ngroup), AD_T, adf_dot2_smem(), st>>>(V, ld, nvec, vpb, adf_cold(nvec, n), x1, x2, part, n, ks);
    // double-float sweeps: the lucky-breakdown threshold of the double-float CGS2 path (1e-11)
    k_adf_dot2_reduce<<<(2 * nvec + 7) / 8, DC_T, 0, st>>>(part, nchunk, nvec, h1, h2, h1d, h2d, H, ldH, ks, 1e-11,
                                                           counter);
}

void launch_adf_dcgs(double2* H, int ldH, const double2* h1, const double2* h2, KState* ks, int j, int fin,
                     cudaStream_t st) {
    k_adf_dcgs<<<1, DC_T, 0, st>>>(H, ldH, h1, h2, ks, j, fin, 1e-11);
}

void launch_adf_update2(const float4* V, size_t ld, int j, const float4* cdf, const float4* ddf, float4* uj,
                        float4* unext, const double2* w, double2* x64, double2* H, int ldH, const double2* h1,
                        const double2* h2, size_t n, KState* ks, cudaStream_t st) {
    const int hb = (j + 1 + AD_W - 1) / AD_W;  // blocks of the rows of H, first
    k_adf_update2<<<hb + adf_update_grid(n), AD_T, 0, st>>>(V, ld, j, adf_cold(j, n), hb, cdf, ddf, uj, unext, w, x64, H,
                                                            ldH, h1, h2, n, ks);
}

void launch_rs_begin(KState* ks, int cyc, cudaStream_t st) { k_rs_begin<<<1, 1, 0, st>>>(ks, cyc); }
void launch_rs_mid(KState* ks, cudaStream_t st) { k_rs_mid<<<1, 1, 0, st>>>(ks); }
void launch_rs_combine(const float4* V, size_t ld, const double2* c, int off, float4* cdf, const KState* ks, int m,
                       double2* y, size_t n, cudaStream_t st) {
    k_rs_coef<<<(m + 255) / 256 > 0 ? (m + 255) / 256 : 1, 256, 0, st>>>(c, cdf, ks, off);
    k_rs_combine<<<(unsigned)((n + 31) / 32), AD_T, 0, st>>>(V, ld, cdf, ks, y, n);
}
void launch_rs_restart(float4* V, size_t ld, int m, const float4* cdf, double2* x64, KState* ks, size_t n, int last,
                       cudaStream_t st) {
    k_rs_restart<<<adf_update_grid(n), AD_T, 0, st>>>(V, ld, m, cdf, x64, ks, n, last);
}

void launch_adf_combine(const float4* V, size_t ld, const double2* c, float4* cdf, const KState* ks, int kmax,
                        double2* y, size_t n, cudaStream_t st) {
    k_adf_coef<<<(kmax + 255) / 256 > 0 ? (kmax + 255) / 256 : 1, 256, 0, st>>>(c, cdf, ks);
    k_adf_combine<<<(unsigned)((n + 31) / 32), AD_T, 0, st>>>(V, ld, cdf, ks, y, n);
}

}  // namespace ovl
