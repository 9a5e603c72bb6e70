"""The FP64 application with a site shared by lanes (device and canonical layout) against one thread per
site, where its units of two or four sites end unevenly and on both sides of the rule that splits the spin
rows (1216 sites).  Both add the same 49 terms per output in another order: a difference of at most
2 x 50 x 2^-53 times the sum of the terms' magnitudes, below 1e-13 of the largest output."""
import numpy as np
import pytest

from gpu_common import KAPPA, torch_c128
from paper_0810_4228_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (3, 3, 3, 2), (3, 5, 3, 4), (4, 4, 4, 18), (5, 5, 5, 10), (4, 4, 4, 20),
                                  (7, 5, 9, 6), (8, 8, 8, 8)])
@pytest.mark.parametrize("bc_t", [-1, 1])
def test_lanes_equal_sites(dims, bc_t):
    import torch
    from paper_0810_4228_gb300 import ovl
    ctx = ovl.Context(dims, bc_t=bc_t)
    ctx.set_gauge(torch_c128(synth.gauge_field(dims, 1.0, 91)))
    x = torch_c128(synth.gaussian_source(dims, 92))
    xn, yn, zn = ctx.empty_native(), ctx.empty_native(), ctx.empty_native()
    ctx.pack(x, xn)
    for fl in (0, ovl.GAMMA5, ovl.DAGGER):
        ref = ctx.apply_Dw(0.3, KAPPA, x, flags=fl | ovl.STENCIL_SITE).cpu().numpy()
        top = np.abs(ref).max()
        assert np.abs(ctx.apply_Dw(0.3, KAPPA, x, flags=fl).cpu().numpy() - ref).max() < 1e-13 * top
        host = ctx.apply_Dw(0.3, KAPPA, x.cpu().numpy(), flags=fl)
        assert np.abs(host - ref).max() < 1e-13 * top
        ctx.apply_Dw(0.3, KAPPA, xn, yn, flags=fl | ovl.NATIVE)
        ctx.apply_Dw(0.3, KAPPA, xn, zn, flags=fl | ovl.NATIVE | ovl.STENCIL_SITE)
        assert float((yn - zn).abs().max()) < 1e-13 * top
    torch.cuda.synchronize()


@pytest.mark.parametrize("shift", [12, -12, 1, 600])
def test_canonical_vectors_that_share_memory(shift):
    """x and y at different places of one buffer: the result is that of separate vectors.  Only the order of the
    sums may differ (through the device layout or not): the bound of the forms above."""
    import torch
    from paper_0810_4228_gb300 import ovl
    dims = (3, 5, 3, 4)
    n = 12 * 3 * 5 * 3 * 4
    ctx = ovl.Context(dims)
    ctx.set_gauge(torch_c128(synth.gauge_field(dims, 1.0, 93)))
    b = torch_c128(synth.gaussian_source(dims, 94))
    ref = ctx.apply_Dw(0.3, KAPPA, b)
    buf = torch.zeros(n + abs(shift), dtype=torch.complex128, device="cuda")
    x, y = (buf[:n], buf[shift:]) if shift > 0 else (buf[-shift:], buf[:n])
    x.copy_(b)
    ctx.apply_Dw(0.3, KAPPA, x, y)
    assert float((y - ref).abs().max()) < 1e-13 * float(ref.abs().max())
