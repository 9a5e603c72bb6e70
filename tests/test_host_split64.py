"""CPU test of the rules by which the cooperative FP64 kernels share a lattice (csrc/split64.h): every unit of
sites belongs to exactly one (block, warp, pass), on both sides of the size where the shared memory of 152
SMs is full, and a launch whose blocks the device does not hold at once is not taken (the per-step kernels
run instead)."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0810_4228_gb300", "csrc")

WRAP = r"""
#include "split64.h"
extern "C" {
void split(int V, int spw, int sms, int* out) {
    const ovl::Split s = ovl::split_units(V, spw, sms);
    out[0] = s.rs, out[1] = s.G, out[2] = s.npass;
}
int fits(int V, int spw, int sms, int per_sm, int coop) {
    return ovl::split_fits(ovl::split_units(V, spw, sms), sms, per_sm, coop != 0);
}
int warps() { return ovl::LW; }
int maxpass() { return ovl::L_MAXPASS; }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("split64")
    (d / "w.cpp").write_text(WRAP)
    so = d / "w.so"
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{CSRC}", str(d / "w.cpp"), "-o", str(so)],
                   check=True)
    return ctypes.CDLL(str(so))


def _split(lib, V, spw, sms):
    o = (ctypes.c_int * 3)()
    lib.split(V, spw, sms, o)
    return o[0], o[1], o[2]


@pytest.mark.parametrize("spw", [2, 4])  # the process (both inputs share a warp), the regeneration
@pytest.mark.parametrize("sms", [1, 76, 148, 152])
def test_units_covered_once(lib, spw, sms):
    for V in (16, 54, 180, 256, 1216, 1218, 1296, 1680, 4096, 13824, 19456, 38912):
        rs, G, npass = _split(lib, V, spw, sms)
        if npass > lib.maxpass():
            continue
        units = -(-V // (spw // rs))
        seen = [b + G * (w + lib.warps() * p) for b in range(G) for w in range(lib.warps()) for p in range(npass)]
        assert sorted(u for u in seen if u < units) == list(range(units)), (V, spw, sms)
        assert G <= sms


def test_size_limits(lib):
    for spw, limit in ((2, 19456), (4, 38912)):
        assert lib.fits(limit, spw, 152, 1, 1) and not lib.fits(limit + spw, spw, 152, 1, 1)


def test_launch_that_does_not_fit(lib):
    for V in (256, 1296, 4096, 19456):
        rs, G, _ = _split(lib, V, 2, 152)
        assert lib.fits(V, 2, 152, 1, 1) and lib.fits(V, 2, 152, 2, 1)
        assert not lib.fits(V, 2, 152, 0, 1)  # one block's shared memory is not to be had
        assert not lib.fits(V, 2, 152, 1, 0)  # no cooperative launches
