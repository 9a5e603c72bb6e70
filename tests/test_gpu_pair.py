"""The pair t = A v, s = A^dag w, alpha = w^dag t on both sides of the rule that goes from the direction split to
one thread per site and stencil (8192 sites), row-grouped and not, against the single applications.

Tolerance: both add the same 49 terms per output in another order, at most 100 roundings of 2^-24 (2^-53) of
the sum of the terms' magnitudes, which here stays below ten times the largest output; alpha is summed to 48
bits or better from the t that is returned, so it has to agree with the FP64 sum over that t to
12 V x 2^-48 of the sum of the terms' magnitudes, itself at most |w| |t|."""
import math

import numpy as np
import pytest

from gpu_common import KAPPA, torch_c128
from paper_0810_4228_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims", [(3, 3, 3, 2), (7, 9, 9, 14), (8, 8, 8, 16), (9, 9, 9, 12), (11, 13, 9, 14), (16, 12, 16, 16)])
def test_pair_equals_single_applications(dims, prec):
    import torch
    from paper_0810_4228_gb300 import ovl
    ctx = ovl.Context(dims)
    ctx.set_gauge(torch_c128(synth.gauge_field(dims, 1.0, 95)))
    mu, f, eps = 0.25, (0, ovl.F32)[prec], (2.0 ** -53, 2.0 ** -24)[prec]
    v, w = (ctx.empty_native(prec) for _ in range(2))
    ctx.pack(torch_c128(synth.gaussian_source(dims, 96)), v, prec)
    ctx.pack(torch_c128(synth.gaussian_source(dims, 97)), w, prec)
    t, s, t1, s1 = (torch.full_like(v, float("nan")) for _ in range(4))
    alpha = ctx.apply_pair(mu, KAPPA, v, w, t, s, prec)
    ctx.apply_Dw(mu, KAPPA, v, t1, flags=ovl.GAMMA5 | ovl.NATIVE | f)
    ctx.apply_Dw(mu, KAPPA, w, s1, flags=ovl.DAGGER | ovl.NATIVE | f)
    for x, y in ((t, t1), (s, s1)):
        assert float((x - y).abs().max()) <= 1000 * eps * float(y.abs().max())
    a, b = w.cpu().numpy().astype(np.complex128), t.cpu().numpy().astype(np.complex128)
    ref = np.vdot(a, b)
    assert abs(alpha - ref) <= 12 * math.prod(dims) * 2.0 ** -48 * np.linalg.norm(a) * np.linalg.norm(b)


@pytest.mark.parametrize("scale", [1.0, 1e-21, 1e21])
@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (9, 9, 9, 12), (16, 12, 16, 16)])
def test_fp32_pair_sums_alpha_in_fp64(dims, scale):
    """Below 155648 sites alpha is an FP64 sum of the FP32 vectors' products in both forms of the kernel: vectors
    whose products leave the FP32 range, and 100 roundings of 2^-53 of the sum of the terms' magnitudes (48 per
    thread, the block's and the grid's trees), which is at most 2 |w| |t|."""
    import torch
    from paper_0810_4228_gb300 import ovl
    ctx = ovl.Context(dims)
    ctx.set_gauge(torch_c128(synth.gauge_field(dims, 1.0, 95)))
    v, w = (ctx.empty_native(1) for _ in range(2))
    ctx.pack(torch_c128(scale * synth.gaussian_source(dims, 98)), v, 1)
    ctx.pack(torch_c128(scale * synth.gaussian_source(dims, 99)), w, 1)
    t, s = (torch.full_like(v, float("nan")) for _ in range(2))
    alpha = ctx.apply_pair(0.25, KAPPA, v, w, t, s, 1)
    a, b = (x.cpu().numpy().astype(np.clongdouble) for x in (w, t))
    ref = (a.conj() * b).sum()
    size = float(np.sqrt((np.abs(a) ** 2).sum()) * np.sqrt((np.abs(b) ** 2).sum()))
    assert abs(complex(alpha - complex(ref))) <= 100 * 2.0 ** -53 * 2 * size


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims", [(18, 21, 20, 22), (32, 31, 32, 34)])
def test_pair_block_orders(dims, prec):
    """Lattices without whole rows per block on both sides of the volume (704512 sites in FP32) where the two kinds of
    block go from one behind the other to alternating: the bounds of the single applications above, and alpha
    against the FP64 sum over the t that is returned."""
    import torch
    from paper_0810_4228_gb300 import ovl
    V, f, eps = math.prod(dims), (0, ovl.F32)[prec], (2.0 ** -53, 2.0 ** -24)[prec]
    ctx = ovl.Context(dims)
    ctx.set_gauge(synth.gauge_field_torch(dims, 1.0, 95))
    gen = torch.Generator("cuda").manual_seed(96)
    v, w = (ctx.empty_native(prec) for _ in range(2))
    for x in (v, w):
        ctx.pack(torch.randn(12 * V, dtype=torch.complex128, device="cuda", generator=gen), x, prec)
    t, s, t1, s1 = (torch.full_like(v, float("nan")) for _ in range(4))
    alpha = ctx.apply_pair(0.25, KAPPA, v, w, t, s, prec)
    ctx.apply_Dw(0.25, KAPPA, v, t1, flags=ovl.GAMMA5 | ovl.NATIVE | f)
    ctx.apply_Dw(0.25, KAPPA, w, s1, flags=ovl.DAGGER | ovl.NATIVE | f)
    for x, y in ((t, t1), (s, s1)):
        assert float((x - y).abs().max()) <= 1000 * eps * float(y.abs().max())
    a, b = (x.to(torch.complex128).flatten() for x in (w, t))
    size = float(torch.linalg.vector_norm(a) * torch.linalg.vector_norm(b))
    assert abs(alpha - complex(torch.vdot(a, b))) <= 12 * V * 2.0 ** -48 * size
