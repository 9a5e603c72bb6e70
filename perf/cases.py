"""Cases that time the library through its public entry points (`paper_0810_4228_gb300.ovl`, `.autograd`).

A case names one call as a user's program makes it: the lattice, the precision and the Krylov size.
`listed()` holds the standing ones, `draw()` more of the same ranges, `prepare()` what the program has
in hand before the call, `run()` the call, `work()` the bytes and operations it cannot do without,
`exact()` the result in plain torch in 64 bits.

Gauge fields are SU(3) links U = exp(i eps H).  The solves take eps = 0.5 (this repository's 4^4
workload), where k = 440 ... 520 steps reach about 1e-13 of the converged result on every lattice of
the ranges without a long set-up of deflation vectors; the operator applications, whose cost does not
depend on eps, take eps = 1.0.
"""
import math

import numpy as np
import torch

from paper_0810_4228_gb300 import autograd, ovl, synth

KAPPA = 0.2          # m_w = -1.5
EPS_SOLVE, EPS_DW = 0.5, 1.0
HOP = 1368           # flop per site of one application of A


def listed():
    return [
        # the smallest call: one application of A on a test lattice, canonical FP64 vectors
        dict(name="dw_f64_4x4x4x4", kind="dw", fmt="f64", dims="4x4x4x4", mu=0.3),
        # the stencil's bandwidth form: FP32, 12-real links, device-layout vectors, far beyond L2
        dict(name="dw_f32_48x48x48x64", kind="dw", fmt="f32", dims="48x48x48x64", mu=0.3),
        # FP32 with full links on a ragged lattice of middling size (A^dag)
        dict(name="dw_f32full_20x18x15x22", kind="dw", fmt="f32full", dims="20x18x15x22", mu=-0.2),
        # the two-sided Lanczos step's pair t = A v, s = A^dag w, alpha = w^dag t
        dict(name="pair_f32_32x32x32x64", kind="pair", fmt="f32", dims="32x32x32x64", mu=0.3),
        # forward and backward of y = A(U, mu) x under autograd (link force, d/dmu, A^dag g)
        dict(name="dw_autograd_24x24x24x24", kind="dwgrad", dims="24x24x24x24", mu=0.2),
        # one source, mixed precision, deflated: the everyday solve on a small lattice
        dict(name="solve_mixed_8x8x8x8_m8", kind="solve", prec="mixed", dims="8x8x8x8", mu=0.3, k=480, m=8),
        # one source, mixed precision, on a lattice of the size production runs use
        dict(name="solve_mixed_16x16x16x32", kind="solve", prec="mixed", dims="16x16x16x32", mu=0.2, k=480, m=0),
        # one source in FP64 throughout, the accuracy reference of the mixed solves
        dict(name="solve_f64_6x6x6x6", kind="solve", prec="f64", dims="6x6x6x6", mu=0.3, k=480, m=0),
        # the Arnoldi method with its basis in double-float
        dict(name="arnoldi_mixed_8x8x8x8", kind="solve", prec="arnoldi", dims="8x8x8x8", mu=0.3, k=450, m=0),
        # a propagator's 12 spin-colour sources on one small lattice
        dict(name="batch_mixed_12_8x8x8x8", kind="batch", dims="8x8x8x8", nrhs=12, mu=0.3, k=480),
        # the benchmark's batch: 12 sources on each of four lattices of uneven sizes
        dict(name="batch_mixed_48_four_lattices", kind="batch", dims="6x6x6x6 8x8x8x8 12x12x12x12 16x16x16x8",
             nrhs=12, mu=0.2, k=480),
        # forward and backward of y = sgn(A(U, mu)) b under autograd
        dict(name="sign_autograd_6x6x6x6", kind="signgrad", dims="6x6x6x6", mu=0.2, k=480),
    ]


def _extents(rng, lo, hi):
    """Four extents of about rng's log-uniform volume in lo..hi: uneven, odd ones among the spatial, even time."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        a = [max(3, round(v ** 0.25 * math.exp(rng.uniform(-0.35, 0.35)))) for _ in range(3)]
        t = max(4, 2 * round(v / (2 * a[0] * a[1] * a[2])))
        if lo <= a[0] * a[1] * a[2] * t <= hi and t <= 4 * max(a):
            return "x".join(str(x) for x in a + [t])


def draw(rng):
    mu = round(rng.uniform(0.05, 0.3), 3)
    k = rng.randint(440, 520)
    kind = rng.choice(["dw", "dw", "pair", "dwgrad", "mixed", "mixed", "f64", "arnoldi", "batch", "batch", "signgrad"])
    if kind == "dw":
        fmt = rng.choice(["f64", "f32", "f32", "f32full"])
        return dict(kind="dw", fmt=fmt, dims=_extents(rng, 256, 1 << 20 if fmt == "f64" else 7 << 20),
                    mu=rng.choice([mu, -mu]))
    if kind == "pair":
        return dict(kind="pair", fmt=rng.choice(["f32", "f32", "f64"]), dims=_extents(rng, 256, 1 << 21), mu=mu)
    if kind == "dwgrad":
        return dict(kind="dwgrad", dims=_extents(rng, 256, 24 ** 4), mu=mu)
    if kind == "mixed":
        dims = _extents(rng, 256, 131072)
        m = rng.choice([0, 4, 8]) if _volume(dims) <= 2048 else 0
        return dict(kind="solve", prec="mixed", dims=dims, mu=mu, k=k, m=m)
    if kind == "f64":
        return dict(kind="solve", prec="f64", dims=_extents(rng, 256, 8192), mu=mu, k=k, m=0)
    if kind == "arnoldi":
        return dict(kind="solve", prec="arnoldi", dims=_extents(rng, 256, 8192), mu=mu, k=rng.randint(200, 450), m=0)
    if kind == "batch":
        dims = " ".join(_extents(rng, 256, 16384) for _ in range(rng.randint(1, 4)))
        return dict(kind="batch", dims=dims, nrhs=rng.randint(1, 12), mu=mu, k=k)
    return dict(kind="signgrad", dims=_extents(rng, 256, 2048), mu=mu, k=k)


# ------------------------------------------------------------------------------ inputs --
def _dims(text):
    return tuple(int(x) for x in text.split("x"))


def _volume(text):
    return math.prod(_dims(text))


def _rng(seed, stream):
    return torch.Generator(device="cuda").manual_seed(1000 * int(seed) + stream)


def _links(dims, eps, seed):
    """SU(3) links [V, 4, 3, 3]: exp(i eps H) on the lattices of the solves; above 2^18 sites, where that
    takes seconds, random SU(3) (Gram-Schmidt on two Gaussian rows, the third their conjugate cross product)."""
    V = math.prod(dims)
    if V <= 1 << 18:
        return synth.gauge_field_torch(dims, eps, 7 * int(seed) + 3)
    g = _rng(seed, 1)
    U = torch.empty((V, 4, 3, 3), dtype=torch.complex128, device="cuda")
    step = 1 << 20
    for s in range(0, V, step):
        u = U[s:s + step]
        a = torch.randn(u.shape[0], 4, 3, dtype=torch.complex128, device="cuda", generator=g)
        b = torch.randn(u.shape[0], 4, 3, dtype=torch.complex128, device="cuda", generator=g)
        a = a / torch.linalg.vector_norm(a, dim=-1, keepdim=True)
        b = b - (a.conj() * b).sum(-1, keepdim=True) * a
        b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
        u[:, :, 0], u[:, :, 1] = a, b
        u[:, :, 2] = torch.linalg.cross(a, b, dim=-1).conj()
    return U


def _spinor(n, seed, stream, dtype=torch.complex128):
    return torch.randn(n, dtype=dtype, device="cuda", generator=_rng(seed, stream))


def prepare(case, seed):
    kind, mu = case["kind"], case["mu"]
    if kind == "batch":
        lats, srcs = [], []
        for j, d in enumerate(case["dims"].split()):
            dims = _dims(d)
            lat = ovl.Context(dims)
            lat.set_gauge(_links(dims, EPS_SOLVE, 16 * seed + j))
            lats.append(lat)
            srcs.append(_spinor((case["nrhs"], 12 * math.prod(dims)), 16 * seed + j, 2))
        batch = ovl.Batch(lats, [case["nrhs"]] * len(lats))
        return dict(case=case, batch=batch, lats=lats, srcs=srcs)
    dims = _dims(case["dims"])
    n = 12 * math.prod(dims)
    lat = ovl.Context(dims)
    eps = EPS_DW if kind in ("dw", "pair", "dwgrad") else EPS_SOLVE
    U = _links(dims, eps, seed)
    lat.set_gauge(U)
    st = dict(case=case, lat=lat)
    if kind == "dw":
        st["x"] = _spinor(n, seed, 2, torch.complex128 if case["fmt"] == "f64" else torch.complex64)
        st["y"] = torch.empty_like(st["x"])
    elif kind == "pair":
        dt = torch.complex128 if case["fmt"] == "f64" else torch.complex64
        st["v"], st["w"] = _spinor(n, seed, 2, dt), _spinor(n, seed, 3, dt)
        st["t"], st["s"] = torch.empty_like(st["v"]), torch.empty_like(st["w"])
    elif kind == "solve":
        st["b"] = _spinor(n, seed, 2)
        if case["m"]:
            lat.deflation_eigs(mu, KAPPA, case["m"], nextra=4)
    else:
        st["U"] = U.requires_grad_()
        st["mu"] = torch.tensor(mu, dtype=torch.float64, device="cuda", requires_grad=True)
        st["x"] = _spinor(n, seed, 2).requires_grad_()
        st["g"] = _spinor(n, seed, 3)
    return st


# -------------------------------------------------------------------------------- runs --
_DW_FLAGS = {"f64": 0, "f32": ovl.NATIVE | ovl.F32, "f32full": ovl.NATIVE | ovl.F32_FULL}
_SOLVE = {"mixed": (ovl.LANCZOS2, ovl.MIXED), "f64": (ovl.LANCZOS2, 0), "arnoldi": (ovl.ARNOLDI, ovl.MIXED)}


def run(state):
    case = state["case"]
    kind, mu = case["kind"], case["mu"]
    if kind == "dw":  # mu < 0 in a case: A^dag at |mu|
        flags = _DW_FLAGS[case["fmt"]] | (ovl.GAMMA5 if mu > 0 else ovl.DAGGER)
        return state["lat"].apply_Dw(abs(mu), KAPPA, state["x"], state["y"], flags=flags)
    if kind == "pair":
        alpha = state["lat"].apply_pair(mu, KAPPA, state["v"], state["w"], state["t"], state["s"],
                                        prec=0 if case["fmt"] == "f64" else 1)
        return [state["t"], state["s"], alpha.real, alpha.imag]
    if kind == "solve":
        method, flags = _SOLVE[case["prec"]]
        return state["lat"].sign_krylov(method, case["k"], mu, KAPPA, state["b"], flags=flags | ovl.OVERLAP)[0]
    if kind == "batch":
        outs, _, _ = state["batch"].solve(case["k"], mu, KAPPA, state["srcs"], flags=ovl.MIXED | ovl.OVERLAP)
        return [row for out in outs for row in out]
    inputs = (state["U"], state["mu"], state["x"])
    if kind == "dwgrad":
        y = autograd.apply_A(*inputs, state["lat"], KAPPA)
    else:
        y = autograd.sign_A(*inputs, state["lat"], KAPPA, case["k"])
    return [y.detach(), *torch.autograd.grad(y, inputs, state["g"])]


def work(case):
    kind, vols = case["kind"], [_volume(d) for d in case["dims"].split()]
    V = sum(vols)
    if kind == "dw":  # links, x, y
        return {"bytes": V * {"f64": 960, "f32": 384, "f32full": 480}[case["fmt"]], "flops": HOP * V}
    if kind == "pair":  # links, v, w, t, s; the dot product on top
        return {"bytes": V * (1344 if case["fmt"] == "f64" else 576), "flops": (2 * HOP + 96) * V}
    if kind == "dwgrad":  # links, x, g in; y, grad_x, grad_U out; two applications, 4 x 2 outer products, d/dmu
        return {"bytes": V * (576 + 4 * 192 + 576), "flops": V * (2 * HOP + 4 * 2 * 4 * 9 * 8 + 500)}
    # a Krylov solve reads the links and its sources and writes its results; its operations are the method's
    n, k = 12 * V, case["k"]
    if kind == "solve":
        m = case["m"]
        if case["prec"] == "arnoldi":  # A v, one Gram-Schmidt pass of 2 x 8 flop per basis element, V c
            flops = k * V * HOP + 8 * n * k * (k + 1) + 8 * n * k
        else:  # A v, A^dag w, two three-term recurrences, three inner products, the combination
            flops = k * (2 * HOP * V + (32 + 16 + 8) * n) + 48 * n * m
        return {"bytes": V * 960, "flops": flops}
    if kind == "batch":
        return {"bytes": V * (576 + 384 * case["nrhs"]), "flops": case["nrhs"] * k * (2 * HOP * V + 56 * n)}
    # signgrad: the forward solve, the process from (b, g), W conj(M), k link forces, V c and W d
    return {"bytes": V * (2 * 576 + 4 * 192), "flops": k * (4 * HOP * V + 128 * n) + 8 * n * k * k + k * V * 2800}


# ------------------------------------------------------- the same in plain torch, 64 bits --
class _Wilson:
    """A = gamma5 D_w(mu) on canonical vectors [..., V, 4, 3] (chiral basis, antiperiodic time)."""

    def __init__(self, dims, U):
        self.dims, self.U = dims, U.detach()
        V = math.prod(dims)
        x = np.indices(dims).reshape(4, -1)
        self.fwd, self.bwd, self.phase = [], [], []
        for nu in range(4):
            to = x.copy()
            to[nu] = (x[nu] + 1) % dims[nu]
            f = np.ravel_multi_index(to, dims)
            b = np.empty(V, dtype=np.int64)
            b[f] = np.arange(V)
            self.fwd.append(torch.from_numpy(f).cuda())
            self.bwd.append(torch.from_numpy(b).cuda())
            ph = np.where((x[nu] == dims[nu] - 1) & (nu == 3), -1.0, 1.0)
            self.phase.append(torch.from_numpy(ph).cuda())  # of the link that leaves each site
        s = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])]
        z = np.zeros((2, 2))
        g = [np.block([[z, -1j * m], [1j * m, z]]) for m in s] + [np.block([[z, np.eye(2)], [np.eye(2), z]])]
        self.gamma = [torch.tensor(m, dtype=torch.complex128, device="cuda") for m in g]
        self.one = torch.eye(4, dtype=torch.complex128, device="cuda")
        self.g5 = torch.tensor([1.0, 1, -1, -1], dtype=torch.float64, device="cuda")[:, None]

    def hops(self, nu, psi):
        """(T_nu^+ psi, T_nu^- psi) without e^{+-mu}."""
        U, ph = self.U[:, nu], self.phase[nu][:, None, None]
        p = torch.einsum("st,xta->xsa", self.one + self.gamma[nu], psi[self.fwd[nu]] * ph)
        q = torch.einsum("st,xta->xsa", self.one - self.gamma[nu], psi * ph)
        b = self.bwd[nu]
        return (U[:, None] @ p[..., None])[..., 0], (U.mH[:, None] @ q[..., None])[..., 0][b]

    def apply(self, psi, mu, derivative=False):
        """gamma5 D_w(mu) psi, or its derivative with respect to mu."""
        psi = psi.reshape(-1, 4, 3)
        out = torch.zeros_like(psi) if derivative else psi.clone()
        for nu in (3,) if derivative else range(4):
            f, b = self.hops(nu, psi)
            cf, cb = (math.exp(mu), math.exp(-mu)) if nu == 3 else (1.0, 1.0)
            out -= KAPPA * (cf * f - cb * b if derivative else cf * f + cb * b)
        return (self.g5 * out).reshape(-1)

    def force(self, x, g, mu):
        """dl/dU of Re <g, A x> summed over the pairs x[q], g[q], as [V, 4, 3, 3]."""
        x, g = x.reshape(-1, self.U.shape[0], 4, 3), self.g5 * g.reshape(-1, self.U.shape[0], 4, 3)
        out = torch.empty_like(self.U)
        for nu in range(4):
            f, ph = self.fwd[nu], self.phase[nu][:, None, None]
            cf, cb = (math.exp(mu), math.exp(-mu)) if nu == 3 else (1.0, 1.0)
            gt = torch.einsum("st,qxta->qxsa", self.one + self.gamma[nu], g)
            gh = torch.einsum("st,qxta->qxsa", self.one - self.gamma[nu], g[:, f])
            out[:, nu] = -KAPPA * ph * (cf * torch.einsum("qxsi,qxsj->xij", gt, x[:, f].conj())
                                        + cb * torch.einsum("qxsi,qxsj->xij", x, gh.conj()))
        return out


def _arnoldi(apply, b, k):
    """Orthonormal basis V [k', N] and the projected k' x k' matrix of K_k(apply, b)."""
    V = torch.empty((k + 1, b.numel()), dtype=torch.complex128, device="cuda")
    H = torch.zeros((k + 1, k), dtype=torch.complex128, device="cuda")
    V[0] = b / torch.linalg.vector_norm(b)
    scale = 0.0
    for j in range(k):
        t = apply(V[j])
        for _ in range(2):
            h = torch.mv(V[:j + 1], t.conj()).conj()
            t = t - torch.mv(V[:j + 1].T, h)
            H[:j + 1, j] += h
        r = float(torch.linalg.vector_norm(t))
        scale = max(scale, float(torch.linalg.vector_norm(H[:j + 1, j])))
        if r <= 1e-12 * scale:
            return V[:j + 1], H[:j + 1, :j + 1]
        H[j + 1, j] = r
        V[j + 1] = t / r
    return V[:k], H[:k, :k]


def _sign(H):
    """sgn of a small matrix: Roberts' iteration S <- (S + S^-1) / 2, determinant-scaled at first."""
    S = H.cpu().numpy()
    for it in range(60):
        X = np.linalg.inv(S)
        c = math.exp(-np.linalg.slogdet(S)[1] / len(S)) if it < 8 else 1.0
        new = 0.5 * (c * S + X / c)
        if it >= 8 and np.linalg.norm(new - S) <= 1e-13 * np.linalg.norm(new):
            break
        S = new
    return torch.from_numpy(new).cuda()


def _sign_times(W, mu, b, k):
    """sgn(A) b by k steps of Arnoldi with Gram-Schmidt applied twice."""
    V, H = _arnoldi(lambda x: W.apply(x, mu), b, k)
    return torch.linalg.vector_norm(b) * torch.mv(V.T, _sign(H)[:, 0])


def _overlap(W, mu, b, k):
    y = _sign_times(W, mu, b, k).reshape(-1, 4, 3)
    return b + (W.g5 * y).reshape(-1)


def _to_sites(dims):
    """Canonical site of every device-layout position: even sites, then odd, both in canonical order."""
    x = np.indices(dims).reshape(4, -1).sum(0) & 1
    return torch.from_numpy(np.concatenate([np.flatnonzero(x == 0), np.flatnonzero(x == 1)])).cuda()


def _from_native(x, dims, at):
    """Device-layout vector (complex64: [6][V][2], complex128: [12][V]) to canonical complex128 [V, 12]."""
    V = math.prod(dims)
    x = x.reshape(6, V, 2).permute(1, 0, 2).reshape(V, 12) if x.dtype == torch.complex64 else x.reshape(12, V).T
    out = torch.empty((V, 12), dtype=torch.complex128, device="cuda")
    out[at] = x.to(torch.complex128)
    return out


def _to_native(x, at, like):
    x = x.reshape(-1, 12)[at]
    x = x.reshape(-1, 6, 2).permute(1, 0, 2) if like == torch.complex64 else x.T
    return x.reshape(-1).contiguous()


def _exact_sign_gradients(W, mu, b, g, k):
    """y = sgn(A) b and the derivatives of Re <g, y>: with R_+- = (A +- i e^u)^-1 they are
    -(1/pi) int e^u sum_+- <R_+-^dag g, dA R_+- b> du, R b and R^dag g each from its own Arnoldi process."""
    nb, ng = torch.linalg.vector_norm(b), torch.linalg.vector_norm(g)
    V, H = _arnoldi(lambda x: W.apply(x, mu), b, k)
    X, K = _arnoldi(lambda x: W.apply(x, -mu), g, k)  # A^dag = gamma5 D_w(-mu)
    y = nb * torch.mv(V.T, _sign(H)[:, 0])
    gb = ng * torch.mv(X.T, _sign(K)[:, 0])
    u = np.arange(-34.0, 34.0, 0.02)  # |A| is about 1: the integrand falls like e^-|u| or faster
    shift = torch.from_numpy(1j * np.concatenate([np.exp(u), -np.exp(u)])).cuda()

    def resolvents(T, s):  # columns (T + s_n)^-1 e_1
        lam, Y = np.linalg.eig(T.cpu().numpy())
        c = np.linalg.solve(Y, np.eye(len(T))[:, 0])
        lam, Y, c = (torch.from_numpy(z).cuda() for z in (lam, Y, c))
        return Y @ (c[:, None] / (lam[:, None] + s))

    a, d = resolvents(H, shift), resolvents(K, -shift)
    M = (shift.abs() * d.conj()) @ a.T
    M *= -0.02 / math.pi * nb * ng
    Z = M.conj().T @ X  # Z_q = sum_p conj(M_pq) x_p
    gU = W.force(V, Z, mu)
    gmu = sum(float((z.conj() * W.apply(v, mu, derivative=True)).sum().real) for z, v in zip(Z, V))
    return [y, gU, torch.tensor(gmu, dtype=torch.float64, device="cuda"), gb]


def exact(case, seed):
    kind, mu = case["kind"], case["mu"]
    if kind == "batch":
        out = []
        for j, d in enumerate(case["dims"].split()):  # the first source of each lattice
            dims = _dims(d)
            W = _Wilson(dims, _links(dims, EPS_SOLVE, 16 * seed + j))
            b = _spinor((case["nrhs"], 12 * math.prod(dims)), 16 * seed + j, 2)
            out += [_overlap(W, mu, b[0], case["k"])] + [None] * (case["nrhs"] - 1)
        return out
    dims = _dims(case["dims"])
    n = 12 * math.prod(dims)
    eps = EPS_DW if kind in ("dw", "pair", "dwgrad") else EPS_SOLVE
    W = _Wilson(dims, _links(dims, eps, seed))
    if kind == "dw":
        if case["fmt"] == "f64":
            return W.apply(_spinor(n, seed, 2), mu)
        at = _to_sites(dims)
        x = _from_native(_spinor(n, seed, 2, torch.complex64), dims, at)
        return _to_native(W.apply(x, mu), at, torch.complex64)
    if kind == "pair":
        dt = torch.complex128 if case["fmt"] == "f64" else torch.complex64
        at = _to_sites(dims)
        v, w = (_from_native(_spinor(n, seed, q, dt), dims, at) for q in (2, 3))
        t, s = W.apply(v, mu), W.apply(w, -mu)
        alpha = (w.reshape(-1).conj() * t).sum()
        return [_to_native(t, at, dt), _to_native(s, at, dt), float(alpha.real), float(alpha.imag)]
    if kind == "solve":
        return _overlap(W, mu, _spinor(n, seed, 2), case["k"])
    x, g = _spinor(n, seed, 2), _spinor(n, seed, 3)
    if kind == "signgrad":
        return _exact_sign_gradients(W, mu, x, g, case["k"])
    gmu = (g.conj() * W.apply(x, mu, derivative=True)).sum().real
    return [W.apply(x, mu), W.force(x, g, mu), gmu, W.apply(g, -mu)]
