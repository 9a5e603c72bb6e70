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


def _force(U, V, Z, dims, mu, bc_t):
    """Sum over the pairs (v_q, Z_q) of the link adjoint of Re <Z_q, A v_q> and of Re <Z_q, dA/dmu v_q>, site by
    site in numpy from Eq. 1.2 (full spinors, all four spins)."""
    s2 = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])]
    o, i2 = np.zeros((2, 2)), np.eye(2)
    gam = [np.block([[o, -1j * s], [1j * s, o]]) for s in s2] + [np.block([[o, i2], [i2, o]])]
    g5 = np.diag([1, 1, -1, -1])
    u = U.reshape(*dims, 4, 3, 3)
    gU, gmu = np.zeros(u.shape, np.complex128), 0.0
    for v, z in zip(V, Z):
        x, g = v.reshape(*dims, 4, 3), np.einsum("st,abcdti->abcdsi", g5, z.reshape(*dims, 4, 3))
        for nu in range(4):
            cf, cb = (np.exp(mu), np.exp(-mu)) if nu == 3 else (1.0, 1.0)
            ph = np.ones(dims)
            if nu == 3:
                ph[..., -1] = bc_t
            xf = np.roll(x, -1, axis=nu)
            gf = np.einsum("st,abcdti->abcdsi", np.eye(4) + gam[nu], g)
            gb = np.roll(np.einsum("st,abcdti->abcdsi", np.eye(4) - gam[nu], g), -1, axis=nu)
            f = -KAPPA * cf * ph[..., None, None] * np.einsum("abcdsi,abcdsj->abcdij", gf, xf.conj())
            b = -KAPPA * cb * ph[..., None, None] * np.einsum("abcdsi,abcdsj->abcdij", x, gb.conj())
            gU[..., nu, :, :] += f + b
            if nu == 3:
                gmu += float((u[..., 3, :, :].conj() * (f - b)).sum().real)
    return gU.reshape(-1, 4, 3, 3), gmu


def _pairs(A, Ah, b, g, k):
    """k steps of two-sided Lanczos from (b, g) (Sec. 4, Eq. 4.2), then the pairs (v_q, Z_q) whose forces add up to
    the derivative of Re <g, sgn(A) b>: -(1/pi) int e^u sum_s <R_s^dag g, dA R_s b> du, R_s = (A + s i e^u)^-1."""
    V, W = [b / np.linalg.norm(b)], []
    zeta = np.vdot(V[0], g)
    W.append(g / zeta)  # zeta = conj(g^dag v_1)
    G = np.zeros((k, k), np.complex128)
    for i in range(k):
        t, s = A @ V[i], Ah @ W[i]
        G[i, i] = np.vdot(W[i], t)
        t, s = t - G[i, i] * V[i], s - np.conj(G[i, i]) * W[i]
        if i:
            t, s = t - G[i - 1, i] * V[i - 1], s - np.conj(G[i, i - 1]) * W[i - 1]
        if i + 1 == k:
            break
        G[i + 1, i] = np.linalg.norm(t)
        G[i, i + 1] = np.vdot(s, t) / G[i + 1, i]
        V.append(t / G[i + 1, i])
        W.append(s / np.conj(G[i, i + 1]))
    h = 0.02
    u = np.arange(-42.0, 42.0, h)
    M, e1 = np.zeros((k, k), np.complex128), np.eye(k)[:, :1]
    for s in (1.0, -1.0):
        sh = 1j * s * np.exp(u)[:, None, None] * np.eye(k)
        a = np.linalg.solve(G + sh, np.broadcast_to(e1, (len(u), k, 1)))[..., 0]
        d = np.linalg.solve(G.conj().T - sh, np.broadcast_to(e1, (len(u), k, 1)))[..., 0]
        M += np.einsum("n,np,nq->pq", np.exp(u), d.conj(), a)
    M *= -h / np.pi * np.linalg.norm(b) * np.conj(zeta)
    return V, M.conj().T @ np.array(W)  # Z_q = sum_p conj(M_pq) w_p


@pytest.mark.parametrize("dims,k,bc_t", [((3, 3, 3, 4), 2, -1), ((3, 3, 3, 4), 7, 1), ((3, 3, 3, 4), 30, -1),
                                         ((2, 2, 2, 4), 5, -1), ((5, 3, 4, 6), 20, 1), ((16, 16, 8, 8), 7, -1)])
def test_sign_grad_equals_restated_sum(dims, k, bc_t):
    """The gradient's force of k pairs in shares (as many as pairs, more pairs than shares and no multiple of
    them, one share on a lattice that fills the SMs alone) against the pairs' single forces added in numpy.
    The two processes differ by rounding, below 1e-10 for k <= 30, and the quadratures by their error, 1e-12;
    1e-8 of the largest entry is far below a share or a pair that is missing or counted twice."""
    import torch
    from oracle import wilson as W
    from paper_0810_4228_gb300 import ovl
    mu, U = 0.2, synth.gauge_field(dims, 0.5, 64)
    b, g = synth.gaussian_source(dims, 65), synth.gaussian_source(dims, 66)
    A = W.a_operator(U, dims, mu, KAPPA, bc_t)
    ref, rmu = _force(U, *_pairs(A, A.conj().T.tocsr(), b, g, k), dims, mu, bc_t)
    ctx = ovl.Context(dims, bc_t=bc_t)
    ctx.set_gauge(torch_c128(U))
    gU = torch.empty((int(np.prod(dims)), 4, 3, 3), dtype=torch.complex128, device="cuda")
    gm, _ = ctx.sign_grad(k, mu, KAPPA, torch_c128(b), torch_c128(g), grad_U=gU)
    assert np.abs(gU.cpu().numpy() - ref).max() < 1e-8 * np.abs(ref).max()
    assert abs(gm - rmu) < 1e-8 * np.linalg.norm(ref)
    gm2, _ = ctx.sign_grad(k, mu, KAPPA, torch_c128(b), torch_c128(g))  # without the links
    assert abs(gm2 - rmu) < 1e-8 * np.linalg.norm(ref)
