"""The double-float regeneration pass (one thread per site, packed FP32x2 arithmetic) against the FP64
regeneration of the same FP32 pass 1, at the sizes where its blocks of 64 sites end unevenly, and its
packed helpers against the scalar double-float arithmetic on the host.

Tolerance: a step's double-float rounding is below 32 x 2^-48 of the vectors' magnitude; over k = 40 steps
of the three-term recurrence, whose rounding errors grow at most by the ratio of the largest vector to the
smallest (below 50 here), 40 x 32 x 2^-48 x 50 = 2.3e-10; typical errors add in quadrature and stay far
below 1e-11, the bound the library states for the two passes' agreement."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from gpu_common import KAPPA, torch_c128
from paper_0810_4228_gb300 import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0810_4228_gb300", "csrc")


@pytest.mark.gpu
@pytest.mark.parametrize("bc_t", [-1, 1])
@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 4), 1), ((3, 3, 3, 4), 3), ((5, 3, 4, 6), 2), ((4, 4, 4, 4), 5)])
def test_regen_df_equals_f64(dims, nrhs, bc_t):
    from paper_0810_4228_gb300 import ovl
    ctx = ovl.Context(dims, bc_t=bc_t)
    ctx.set_gauge(torch_c128(synth.gauge_field(dims, 0.5, 71)))
    b = torch_c128(synth.gaussian_source(dims, 72, nrhs=nrhs))
    other = ovl.Context((4, 2, 2, 4), bc_t=bc_t)
    other.set_gauge(torch_c128(synth.gauge_field((4, 2, 2, 4), 0.5, 73)))
    ob = torch_c128(synth.gaussian_source((4, 2, 2, 4), 74, nrhs=1))
    bt = ovl.Batch([ctx, other], [nrhs, 1])
    for minb in (3, 4):
        bt.set_tuning(128, minb)
        for k in (1, 2, 3, 40):
            yd = bt.solve(k, 0.3, KAPPA, [b, ob], flags=ovl.MIXED)[0]
            y6 = bt.solve(k, 0.3, KAPPA, [b, ob], flags=ovl.MIXED | ovl.PASS2_F64)[0]
            for u, v in zip(yd, y6):
                err = np.linalg.norm((u - v).cpu().numpy()) / np.linalg.norm(v.cpu().numpy())
                assert err < 1e-11, (k, minb, err)
    bt.close()


WRAP = r"""
#include "df32.cuh"
using namespace ovl;
static float2 at(const float* p, int i) { return make_float2(p[2 * i], p[2 * i + 1]); }
extern "C" void pair(const float* v, int n, const float* sg, float* o, float* ref) {
    // packed: (s, e) = sum_k a_k b_k, then a signed pair added, then renormalised
    dfacc2 A;
    for (int k = 0; k < n; ++k) {
        const float* q = v + 8 * k;
        if (k == 0) dfacc2_first(A, at(q, 0), at(q, 1), at(q, 2), at(q, 3));
        else dfacc2_add(A, at(q, 0), at(q, 1), at(q, 2), at(q, 3));
    }
    dfacc2_add_signed(A, make_float2(sg[0], sg[1]), at(v, 0), at(v, 1));
    const dfacc2 r = dfacc2_value(A);
    o[0] = r.s.x, o[1] = r.s.y, o[2] = r.e.x, o[3] = r.e.y;
    for (int h = 0; h < 2; ++h) {  // the same, one half at a time
        dfacc S;
        for (int k = 0; k < n; ++k) {
            const float* q = v + 8 * k + h;
            if (k == 0) dfacc_first(S, df(q[0], q[2]), df(q[4], q[6]), false);
            else dfacc_add(S, df(q[0], q[2]), df(q[4], q[6]), false);
        }
        const df z = df_add_lazy(df(S.s, S.e), df(sg[h] * v[h], sg[h] * v[2 + h]));
        const df w = df_fast2sum(z.hi, z.lo);
        ref[h] = w.hi, ref[2 + h] = w.lo;
    }
}
"""


@pytest.mark.parametrize("n", [1, 2, 6])
def test_packed_equals_scalar(tmp_path, n):
    """Each half of the packed operations gives the scalar operation's pair: leading parts equal, trailing
    parts to the rounding of their own sum (two additions may be ordered differently)."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "w.cu"
    src.write_text(WRAP)
    so = tmp_path / "w.so"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "-I", CSRC, "-shared",
                    "-Xcompiler", "-fPIC,-ffp-contract=off", str(src), "-o", str(so)], check=True)
    fn = ctypes.CDLL(str(so)).pair
    rng = np.random.default_rng(5)
    P = ctypes.POINTER(ctypes.c_float)
    for _ in range(400):
        hi = (rng.standard_normal((n, 2, 2)) * 10.0 ** rng.integers(-6, 7, (n, 2, 2))).astype(np.float32)
        lo = (hi * rng.uniform(-3e-8, 3e-8, hi.shape)).astype(np.float32)
        v = np.stack([hi, lo], axis=2).reshape(n, 8)[:, [0, 1, 2, 3, 4, 5, 6, 7]].astype(np.float32).copy()
        sg = rng.choice([-1.0, 1.0], 2).astype(np.float32)
        o, ref = np.zeros(4, np.float32), np.zeros(4, np.float32)
        fn(v.ctypes.data_as(P), n, sg.ctypes.data_as(P), o.ctypes.data_as(P), ref.ctypes.data_as(P))
        scale = np.abs(hi[:, 0] * hi[:, 1]).astype(np.float64).sum(0) + np.abs(hi[0, 0])
        full = o[:2].astype(np.float64) + o[2:].astype(np.float64)
        rfull = ref[:2].astype(np.float64) + ref[2:].astype(np.float64)
        assert np.all(np.abs(full - rfull) <= 4 * 2.0 ** -48 * scale), (o, ref)
