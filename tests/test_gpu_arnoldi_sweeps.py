"""The double-float Arnoldi's two sweeps per step (delayed Gram-Schmidt) against its four classical sweeps
(OVL_ARNOLDI_CGS2), at the sizes where their tiles end unevenly: vectors that are no multiple of the 128
staged or the 512 summed elements, vector counts around the warps' rounds of 4 x 8, more vectors than one
staging of 512 coefficients, and a basis beyond the part that the sweeps keep in L2.

Tolerance: both build the process to the basis's double-float rounding, 2^-48 = 3.6e-15 of a vector, and
Arnoldi does not amplify it beyond the number of steps: 600 x 3.6e-15 = 2.2e-12 at the largest k."""
import pytest

from gpu_common import KAPPA, rel, torch_c128
from paper_0810_4228_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ks", [((3, 3, 3, 2), (1, 31)), ((3, 5, 3, 4), (32, 33, 65)), ((4, 4, 4, 4), (8, 9, 127)),
                                     ((5, 3, 7, 6), (130, 600)), ((9, 8, 7, 8), (150,))])
def test_two_sweeps_match_four(dims, ks):
    from paper_0810_4228_gb300 import ovl
    ctx = ovl.Context(dims)
    ctx.set_gauge(torch_c128(synth.gauge_field(dims, 0.5, 91)))
    b = torch_c128(synth.gaussian_source(dims, 92))
    for k in ks:
        y, i1 = ctx.sign_krylov(ovl.ARNOLDI, k, 0.3, KAPPA, b, flags=ovl.MIXED)
        z, i2 = ctx.sign_krylov(ovl.ARNOLDI, k, 0.3, KAPPA, b, flags=ovl.MIXED | ovl.ARNOLDI_CGS2)
        assert i1["status"] == i2["status"] == 0 and i1["k_used"] == i2["k_used"]
        assert rel(y.cpu().numpy(), z.cpu().numpy()) < 2.2e-12, k
