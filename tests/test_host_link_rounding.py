"""CPU test of the two roundings of the FP32 link product (csrc/ovl_common.cuh): mul_link_pf and
mul_link_dag_pf (the batch's FP32 pass) form every product first, to the bit as numpy's FP32 arithmetic does
in the same order; mul_link and mul_link_dag chain fused multiply-adds.  Both are functions of one name and
one meaning each, in every translation unit.  Against FP64 each stays within the bound of six products and
their sums, 8 x 2^-24 of the sum of the terms' magnitudes."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0810_4228_gb300", "csrc")

WRAP = r"""
#include "ovl_common.cuh"
using namespace ovl;
extern "C" void link(const float* u, const float* h, float* o, int dag, int pf) {
    Link<float> U;
    Half<float> H, O;
    for (int e = 0; e < 9; ++e) U.u[e / 3][e % 3] = mk(u[2 * e], u[2 * e + 1]);
    for (int e = 0; e < 6; ++e) H.h[e / 3][e % 3] = mk(h[2 * e], h[2 * e + 1]);
    if (dag) pf ? mul_link_dag_pf(U, H, O) : mul_link_dag(U, H, O);
    else pf ? mul_link_pf(U, H, O) : mul_link(U, H, O);
    for (int e = 0; e < 6; ++e) o[2 * e] = O.h[e / 3][e % 3].r, o[2 * e + 1] = O.h[e / 3][e % 3].i;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if not nvcc:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("link")
    (d / "w.cu").write_text(WRAP)
    subprocess.run([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC,-ffp-contract=off", "-I", CSRC,
                    "-gencode", "arch=compute_103a,code=sm_103a", str(d / "w.cu"), "-o", str(d / "w.so")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


def _products_first(U, h, dag):
    f = np.float32
    o = np.zeros((2, 3, 2), f)
    for s in range(2):
        for a in range(3):
            for k in range(3):
                b = U[k, a] if dag else U[a, k]
                br, bi, cr, ci = f(b.real), f(b.imag), f(h[s, k].real), f(h[s, k].imag)
                if dag:
                    re, im = f(br * cr) + f(bi * ci), f(br * ci) - f(bi * cr)
                else:
                    re, im = f(br * cr) - f(bi * ci), f(br * ci) + f(bi * cr)
                o[s, a, 0] = re if k == 0 else f(o[s, a, 0] + re)
                o[s, a, 1] = im if k == 0 else f(o[s, a, 1] + im)
    return o


@pytest.mark.parametrize("dag", [0, 1])
def test_link_product_roundings(lib, dag):
    rng = np.random.default_rng(5)
    differ = 0
    for _ in range(200):
        U = (rng.normal(size=(3, 3)) + 1j * rng.normal(size=(3, 3))).astype(np.complex64)
        h = (rng.normal(size=(2, 3)) + 1j * rng.normal(size=(2, 3))).astype(np.complex64)
        got = []
        for pf in (0, 1):
            o = np.zeros((2, 3, 2), np.float32)
            lib.link(U.ctypes.data_as(ctypes.c_void_p), h.ctypes.data_as(ctypes.c_void_p),
                     o.ctypes.data_as(ctypes.c_void_p), dag, pf)
            got.append(o)
        assert np.array_equal(got[1], _products_first(U, h, dag))
        M = (U.conj().T if dag else U).astype(np.complex128)
        ref, mag = h.astype(np.complex128) @ M.T, np.abs(h) @ np.abs(M).T
        for o in got:
            z = o[..., 0].astype(np.float64) + 1j * o[..., 1]
            assert np.all(np.abs(z - ref) <= 8 * 2.0 ** -24 * 2 * mag)
        differ += not np.array_equal(*got)
    assert differ > 100  # the two forms are two forms
