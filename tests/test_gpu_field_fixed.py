"""The FP64 form's solve in 64-bit fixed point keeps what FP64 cycles give: the
residual norms in FP64."""
import pytest

from gpu_util import small_phys
from paper_2307_01797_gb300 import itokmc
from test_gpu_field_forms import rel_residual

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ions", [(16, 3), (32, 1000), (64, 77777)])
def test_norms_are_fp64(n, ions):
    # a uniform charge: the sum of equal squares rounds the same way all along,
    # up to 2^-24 per term of a partial sum in FP32.  In FP64: 2^-53 per term
    # and level of the sum (below 1e-14), and the rounding of the potential
    # to FP64, 12 * 2^-53 |phi| per cell against a residual of 1e-3 b or more
    # with |phi| < b n^2 / 8 (below 1e-9 at n = 64 if all signs agreed; they do
    # not: 2^18 cells of either sign leave 2^-9 of it)
    import torch
    ph = small_phys(n, E0=0.0, mg_rtol=0.2)
    rho = torch.full((n ** 3,), ions << 30, dtype=torch.int64, device="cuda")
    phi = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    E = torch.empty(3 * n ** 3, dtype=torch.float64, device="cuda")
    _, rel = itokmc.itokmc_field_solve_noalloc(itokmc.make_config(ph, 1), rho, phi, E)
    assert 1e-3 < rel <= 0.2
    want = rel_residual(phi.cpu().numpy(), rho.cpu().numpy(), ph)
    assert abs(rel - want) <= 1e-11 * want
