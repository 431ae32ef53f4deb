"""The FP64 form's solve in 64-bit fixed point keeps what FP64 cycles give: the
residual norms in FP64, a scale per realization, at least the 53 bits of a
double for the largest potential, whatever the start guess."""
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
    # and level of the sum (below 1e-14), and the rounding of the potential to
    # FP64: 12 * 2^-53 |phi| per cell, |phi| < b n^2 / 8, of either sign over
    # n^3 cells whose residual is 1e-2 b or more (below 2e-12 at n = 64)
    import torch
    ph = small_phys(n, E0=0.0, mg_rtol=0.2)
    rho = torch.full((n ** 3,), ions << 30, dtype=torch.int64, device="cuda")
    phi = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    E = torch.empty(3 * n ** 3, dtype=torch.float64, device="cuda")
    _, rel = itokmc.itokmc_field_solve_noalloc(itokmc.make_config(ph, 1), rho, phi, E)
    assert 1e-3 < rel <= 0.2
    want = rel_residual(phi.cpu().numpy(), rho.cpu().numpy(), ph)
    assert abs(rel - want) <= 1e-11 * want


def bits_held(phi):
    """Bits between the leading one of the largest |phi| and the last one set
    in any value of at least a quarter of it."""
    a = np.abs(phi)
    m, e = np.frexp(a[a >= a.max() / 4])
    mant = (m * 2.0 ** 53).astype(np.int64)
    last = min(int(ee) - 53 + (int(v) & -int(v)).bit_length() - 1 for v, ee in zip(mant, e))
    return int(np.frexp(a.max())[1]) - last


@pytest.mark.parametrize("n", [16, 64])
def test_a_weak_member_beside_a_strong_one(n):
    # the strong member's potential is 2e4 times and more the weak ones'; FP64
    # cycles hold 53 bits of each (54 and 55 where values of the next lower
    # binades show), one scale for all leaves 39 to 42
    ph = small_phys(n, E0=0.0)
    H = itokmc.Handle(itokmc.make_config(ph, 100, realizations=3))
    pos = np.concatenate([charges("cloud", n, 0), np.full(n ** 3, 10 ** 6), charges("cloud", n, 1)])
    H.itokmc_set_ions(pos, np.zeros_like(pos))
    H.itokmc_solve_field()
    phi = H.itokmc_read_densities(itokmc.PHI, -1).reshape(3, -1)
    rho = H.itokmc_read_densities(itokmc.RHO, -1).reshape(3, -1)
    for r in range(3):
        assert rel_residual(phi[r], rho[r], ph) <= TOL
        assert bits_held(phi[r]) >= 53
    H.close()


def bits_of_largest(phi):
    """Bits between the leading one of the largest |phi| and the last one set
    in any value: the step in which the potential is held (n^3 values do not
    all have a last bit of zero; a single value does every other time)."""
    m, e = np.frexp(np.abs(phi[phi != 0.0]))
    mant = (m * 2.0 ** 53).astype(np.int64)
    low = np.log2((mant & -mant).astype(np.float64)).astype(np.int64)
    return int(e.max() - (e.astype(np.int64) - 53 + low).min())


@pytest.mark.parametrize("rtol", [1e-3, 1e-10])
@pytest.mark.parametrize("kind", ["point", "corner", "cloud"])
@pytest.mark.parametrize("n", [16, 64])
def test_the_largest_potential_has_53_bits(n, kind, rtol):
    # the bound from which a scale is taken is 2^12 above a single cell's potential
    ph = small_phys(n, E0=0.0, mg_rtol=rtol)
    H = itokmc.Handle(itokmc.make_config(ph, 100))
    pos, none = charges(kind, n, 1), np.zeros(n ** 3, np.int64)
    H.itokmc_set_ions(pos, none)
    H.itokmc_solve_field()
    phi = H.itokmc_read_densities(itokmc.PHI)
    assert rel_residual(phi, H.itokmc_read_densities(itokmc.RHO), ph) <= 1.02 * rtol
    assert bits_of_largest(phi) >= 53
    # the same charge again: the guess needs no cycle and stays as it is
    H.itokmc_solve_field()
    if H.itokmc_get_stats()["mg_cycles"] == 0:
        assert np.array_equal(H.itokmc_read_densities(itokmc.PHI), phi)
    # a weaker charge: the guess' leading bits are not the solution's
    H.itokmc_set_ions(charges("corner", n, 1), none)
    H.itokmc_solve_field()
    phi = H.itokmc_read_densities(itokmc.PHI)
    assert rel_residual(phi, H.itokmc_read_densities(itokmc.RHO), ph) <= 1.02 * rtol
    assert bits_of_largest(phi) >= 53
    H.close()


@pytest.mark.parametrize("factor", [30, 10 ** 6])
@pytest.mark.parametrize("n,graph", [(16, 0), (64, 0), (16, 1)])
def test_a_charge_that_jumps_between_steps(n, graph, factor):
    # steps take their scale from the extrapolated potential
    ph = small_phys(n, E0=0.0)
    H = itokmc.Handle(itokmc.make_config(ph, 10000, graph_step=graph))
    c = (np.arange(8) + 0.5) * (ph["hi"][0] - ph["lo"][0]) / 8 + ph["lo"][0]
    H.itokmc_set_particles(c, c, c, np.ones(8, np.uint32))
    none = np.zeros(n ** 3, np.int64)
    for scale in (1, factor, 1):
        H.itokmc_set_ions(scale * charges("cloud", n, 2), none)
        for _ in range(3):
            H.itokmc_step(1)
            rho = H.itokmc_read_densities(itokmc.RHO)
            assert rel_residual(H.itokmc_read_densities(itokmc.PHI), rho, ph) <= TOL
    H.close()
