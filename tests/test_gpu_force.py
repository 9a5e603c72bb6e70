"""The half-spinor link force against the oracle's derivative of A on lattices where blocks of 32 sites end
unevenly and where the pairs' shares are uneven (k not a multiple of the shares).  FP64: 200 products per
entry, 1e-12 of the largest entry; the mu derivative is a sum over 4 V 9 terms, 1e-12 of their magnitude."""
import numpy as np
import pytest

from gpu_common import KAPPA, torch_c128
from oracle import frechet as Fr
from paper_0810_4228_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (3, 3, 3, 2), (3, 5, 3, 4)])
@pytest.mark.parametrize("bc_t", [-1])
def test_dw_grad_entries(dims, bc_t):
    import torch
    from paper_0810_4228_gb300 import ovl
    mu, V = 0.3, int(np.prod(dims))
    U, x, g = synth.gauge_field(dims, 1.0, 61), synth.gaussian_source(dims, 62), synth.gaussian_source(dims, 63)
    ctx = ovl.Context(dims, bc_t=bc_t)
    ctx.set_gauge(torch_c128(U))
    gU = torch.empty((V, 4, 3, 3), dtype=torch.complex128, device="cuda")
    _, gm = ctx.dw_grad(mu, KAPPA, torch_c128(x), torch_c128(g), gU)
    _, gm0 = ctx.dw_grad(mu, KAPPA, torch_c128(x), torch_c128(g))  # without the links
    got = gU.cpu().numpy()
    rng = np.random.default_rng(3)
    for _ in range(12):  # single entries: dl = Re conj(g_U) dU
        dU = np.zeros_like(U)
        e = (rng.integers(V), rng.integers(4), rng.integers(3), rng.integers(3))
        dU[e] = 1.0
        re = np.real(np.vdot(g, Fr.dA_dU_apply(U, dU, dims, mu, KAPPA, x)))
        dU[e] = 1j
        im = np.real(np.vdot(g, Fr.dA_dU_apply(U, dU, dims, mu, KAPPA, x)))
        assert abs(got[e] - (re + 1j * im)) < 1e-12 * np.abs(got).max()
    ref = np.real(np.vdot(g, Fr.dA_dmu(U, dims, mu, KAPPA) @ x))
    size = np.linalg.norm(g) * np.linalg.norm(x)
    assert abs(gm - ref) < 1e-12 * size and abs(gm0 - ref) < 1e-12 * size


@pytest.mark.parametrize("k", [2, 7, 30])
def test_sign_grad_shares(k):
    """The force of k pairs split into shares: equal to the sum of the pairs' single forces through the
    gradient's own linearity in g (g and 2 g give the same process up to scale)."""
    import torch
    from paper_0810_4228_gb300 import ovl
    dims = (3, 3, 3, 4)
    V = int(np.prod(dims))
    ctx = ovl.Context(dims)
    ctx.set_gauge(torch_c128(synth.gauge_field(dims, 0.5, 64)))
    b, g = torch_c128(synth.gaussian_source(dims, 65)), torch_c128(synth.gaussian_source(dims, 66))
    out = []
    for f in (1.0, 2.0):  # a power of two: every quantity of the second run is the first's times 2 exactly
        gU = torch.empty((V, 4, 3, 3), dtype=torch.complex128, device="cuda")
        gm, _ = ctx.sign_grad(k, 0.2, KAPPA, b, f * g, grad_U=gU)
        out.append((gm, gU))
    assert abs(out[1][0] - 2 * out[0][0]) <= 1e-12 * abs(out[1][0])
    assert float((out[1][1] - 2 * out[0][1]).abs().max()) <= 1e-12 * float(out[1][1].abs().max())
