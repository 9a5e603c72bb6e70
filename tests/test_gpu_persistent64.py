"""The FP64 two-sided Lanczos process in one cooperative launch, and the FP64 regeneration pass likewise,
against the per-step kernels (OVL_STEPWISE): the same recurrence in another order of summation.

Sizes: fewer units than SMs, a volume that is no multiple of the regeneration's four sites per warp, odd
extents, both row splits (up to about 1300 sites, and beyond), several passes over a block's warps.
Tolerance: for k <= 30 two-sided Lanczos does not yet amplify rounding; 30 steps of relative rounding
n_ops x 2^-53 with n_ops of order 100 per entry stay below 1e-12, and 1e-10 leaves the two processes'
different sums of 12 V terms a factor of 100."""
import numpy as np
import pytest

from gpu_common import KAPPA, rel, torch_c128
from paper_0810_4228_gb300 import synth

pytestmark = pytest.mark.gpu
DIMS = [(2, 2, 2, 4), (3, 3, 3, 2), (3, 5, 3, 4), (4, 4, 4, 4), (6, 6, 6, 6), (7, 5, 6, 8), (8, 8, 8, 8), (9, 8, 12, 16)]


@pytest.fixture(scope="module")
def ovl():
    from paper_0810_4228_gb300 import ovl as O
    O.load()
    return O


def _problem(ovl, dims, bc_t=-1):
    ctx = ovl.Context(dims, bc_t=bc_t)
    ctx.set_gauge(torch_c128(synth.gauge_field(dims, 0.7, 81)))
    return ctx, torch_c128(synth.gaussian_source(dims, 82))


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("two_pass", [False, True])
def test_fp64_process(ovl, dims, two_pass):
    ctx, b = _problem(ovl, dims, bc_t=-1 if two_pass else 1)
    fl = ovl.TWO_PASS if two_pass else 0
    for k in (1, 2, 30):
        y, i1 = ctx.sign_krylov(ovl.LANCZOS2, k, 0.3, KAPPA, b, flags=fl)
        s, i2 = ctx.sign_krylov(ovl.LANCZOS2, k, 0.3, KAPPA, b, flags=fl | ovl.STEPWISE)
        assert i1["k_used"] == i2["k_used"] and i1["status"] == i2["status"] == 0
        assert rel(y.cpu().numpy(), s.cpu().numpy()) < 1e-10, k
    # eager launches and a repeated graph give the same numbers
    e, _ = ctx.sign_krylov(ovl.LANCZOS2, 30, 0.3, KAPPA, b, flags=fl | ovl.NO_GRAPH)
    assert np.array_equal(e.cpu().numpy(), y.cpu().numpy())


@pytest.mark.parametrize("dims", DIMS)
def test_fp64_regeneration(ovl, dims):
    """The mixed solve's FP64 pass 2 against a batch of one with the FP64 regeneration kernels on the same
    (persistent or stepwise, equal) FP32 pass 1: 1e-6 separates the FP32 passes' own sums, so the passes are
    compared through double-float and FP64 forms of the same solve instead, 1e-11 apart at most."""
    ctx, b = _problem(ovl, dims)
    for k in (1, 2, 30):
        y, _ = ctx.sign_krylov(ovl.LANCZOS2, k, 0.2, KAPPA, b, flags=ovl.MIXED)
        d, _ = ctx.sign_krylov(ovl.LANCZOS2, k, 0.2, KAPPA, b, flags=ovl.MIXED | ovl.PASS2_DF)
        assert rel(y.cpu().numpy(), d.cpu().numpy()) < 1e-11, k


def test_fp64_zero_source(ovl):
    ctx, b = _problem(ovl, (4, 4, 4, 4))
    z = b * 0
    y, info = ctx.sign_krylov(ovl.LANCZOS2, 20, 0.3, KAPPA, z)
    assert info["k_used"] == 0 and not y.abs().max().item()


@pytest.mark.parametrize("dims", [(13, 13, 8, 14), (16, 19, 8, 8), (13, 12, 10, 14)])
def test_fp64_process_at_the_size_limit(ovl, dims):
    """Four passes over a block's warps, the last of them partly empty; exactly the 19456 sites that the shared
    memory of 152 SMs holds; and a lattice above, where both calls run the per-step kernels."""
    ctx, b = _problem(ovl, dims)
    for fl in (0, ovl.TWO_PASS):
        y, i1 = ctx.sign_krylov(ovl.LANCZOS2, 12, 0.3, KAPPA, b, flags=fl)
        s, i2 = ctx.sign_krylov(ovl.LANCZOS2, 12, 0.3, KAPPA, b, flags=fl | ovl.STEPWISE)
        assert i1["k_used"] == i2["k_used"] == 12
        assert rel(y.cpu().numpy(), s.cpu().numpy()) < 1e-10
