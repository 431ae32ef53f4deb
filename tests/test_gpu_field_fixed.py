"""The FP64 form's solve in 64-bit fixed point keeps what FP64 cycles give: the
residual norms in FP64, a scale per realization, at least the 53 bits of a
double for the largest potential, start guesses far from the solution."""
import numpy as np
import pytest

from gpu_util import small_phys
from paper_2307_01797_gb300 import itokmc
from test_gpu_field_forms import TOL, charges, rel_residual

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


@pytest.mark.parametrize("n", [16, 64])
def test_a_weak_member_beside_a_strong_one(n):
    # the strong member's potential is 1e11 and more times the weak one's
    ph = small_phys(n, E0=0.0)
    H = itokmc.Handle(itokmc.make_config(ph, 100, realizations=3))
    pos = np.concatenate([charges("corner", n, 0), np.full(n ** 3, 3 * 10 ** 9), charges("point", n, 0)])
    H.itokmc_set_ions(pos, np.zeros_like(pos))
    H.itokmc_solve_field()
    phi = H.itokmc_read_densities(itokmc.PHI, -1).reshape(3, -1)
    rho = H.itokmc_read_densities(itokmc.RHO, -1).reshape(3, -1)
    for r in range(3):
        assert rel_residual(phi[r], rho[r], ph) <= TOL
    H.close()


def bits_held(phi):
    """Bits between the leading one of the largest |phi| and the last one set
    in any value of at least a quarter of it."""
    a = np.abs(phi)
    m, e = np.frexp(a[a >= a.max() / 4])
    mant = (m * 2.0 ** 53).astype(np.int64)
    last = min(int(ee) - 53 + (int(v) & -int(v)).bit_length() - 1 for v, ee in zip(mant, e))
    return int(np.frexp(a.max())[1]) - last


@pytest.mark.parametrize("rtol", [1e-3, 1e-10])
@pytest.mark.parametrize("kind", ["point", "corner", "cloud"])
@pytest.mark.parametrize("n", [16, 64])
def test_the_largest_potential_has_53_bits(n, kind, rtol):
    ph = small_phys(n, E0=0.0, mg_rtol=rtol)
    H = itokmc.Handle(itokmc.make_config(ph, 100))
    H.itokmc_set_ions(charges(kind, n, 1), np.zeros(n ** 3, np.int64))
    H.itokmc_solve_field()
    phi = H.itokmc_read_densities(itokmc.PHI)
    assert rel_residual(phi, H.itokmc_read_densities(itokmc.RHO), ph) <= 1.02 * rtol
    # values of the next lower binades have 53 bits from a lower leading one:
    # FP64 cycles end at 53 to 55 here
    assert bits_held(phi) >= 53
    H.close()


@pytest.mark.parametrize("ions", [1000, 1200, 1400, 1700, 1999])
def test_a_charge_that_changes_sign(ions):
    # a uniform charge reaches the bound from which the scale is taken, and
    # the error of the last potential is twice it
    n = 32
    ph = small_phys(n, E0=0.0)
    H = itokmc.Handle(itokmc.make_config(ph, 100))
    c, z = np.full(n ** 3, ions, np.int64), np.zeros(n ** 3, np.int64)
    cycles = []
    for pos, neg in ((c, z), (z, c), (c, z)):
        H.itokmc_set_ions(pos, neg)
        H.itokmc_solve_field()
        assert rel_residual(H.itokmc_read_densities(itokmc.PHI), H.itokmc_read_densities(itokmc.RHO), ph) <= TOL
        cycles.append(H.itokmc_get_stats()["mg_cycles"])
    assert max(cycles) <= cycles[0] + 1
    H.close()
