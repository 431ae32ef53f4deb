"""The multigrid at the edges of its kernels: the coarse kernel's starting
levels (8^3, 16^3, 32^3), one tile and several tiles of the fused sweeps (64^3,
128^3), one and three realizations, odd and uneven sweep counts; and the FP64
form's integer cycles where their scale is hard: no applied field with a single
charged cell, a charge far below the applied potential, a start guess beyond
the integers' range (the FP64 cycles take over).

The checked property is the solver's own: the residual of the discrete
equation, formed here in FP64 from the returned potential, is at most mg_rtol
= 1e-10 of the right-hand side.  The allowance of 2e-12 is for the rounding of
the potential to FP64 and of the residual's evaluation: 12 operations of 2^-53
|phi| per cell against |b|, below 1e-13 relative here, and the norm's FP32
partial sums (2^-24 of the norm, 6e-18)."""
import numpy as np
import pytest

from gpu_util import small_phys
from oracle import poisson
from paper_2307_01797_gb300 import itokmc

pytestmark = pytest.mark.gpu
TOL = 1.02e-10


def rel_residual(phi, rho, ph):
    n = ph["n"]
    h = (ph["hi"][0] - ph["lo"][0]) / n
    top = ph["E0"] * (ph["hi"][2] - ph["lo"][2])
    phi = phi.reshape(n, n, n)
    # the boundary values are folded into b: apply the homogeneous operator
    b = poisson.rhs(rho, n, h, 10, top)
    r = b - poisson.apply_operator(phi, h, 0.0)
    return np.linalg.norm(r) / np.linalg.norm(b)


def charges(kind, n, seed):
    rng = np.random.default_rng(seed)
    pos = np.zeros(n ** 3, np.int64)
    if kind == "point":
        pos[(n // 2 * n + n // 3) * n + n // 4] = 1000
    elif kind == "corner":
        pos[0] = 7
    else:
        pos = rng.poisson(50.0, n ** 3).astype(np.int64)
        pos.reshape(n, n, n)[: n // 2] *= 3
    return pos


@pytest.mark.parametrize("precision", [itokmc.FP64, itokmc.MIXED])
@pytest.mark.parametrize("n,R,nu", [(8, 1, (2, 2)), (16, 3, (2, 2)), (32, 1, (1, 2)), (64, 1, (2, 2)),
                                    (64, 3, (3, 1)), (128, 1, (4, 3))])
def test_residual_reaches_the_tolerance(n, R, nu, precision):
    ph = small_phys(n)
    H = itokmc.Handle(itokmc.make_config(ph, 100, realizations=R, precision=precision, mg_nu1=nu[0], mg_nu2=nu[1]))
    pos = np.concatenate([charges("cloud", n, 5 + r) for r in range(R)])
    neg = np.concatenate([charges("cloud", n, 50 + r)[::-1] for r in range(R)])
    H.itokmc_set_ions(pos, neg)
    H.itokmc_solve_field()
    phi = H.itokmc_read_densities(itokmc.PHI, -1).reshape(R, -1)
    rho = H.itokmc_read_densities(itokmc.RHO, -1).reshape(R, -1)
    for r in range(R):
        assert rel_residual(phi[r], rho[r], ph) <= TOL
    H.close()


@pytest.mark.parametrize("kind,E0", [("point", 0.0), ("corner", 0.0), ("corner", 1.5e6)])
@pytest.mark.parametrize("n", [16, 64])
def test_localised_charge(n, kind, E0):
    ph = small_phys(n, E0=E0)
    H = itokmc.Handle(itokmc.make_config(ph, 100))
    H.itokmc_set_ions(charges(kind, n, 1), np.zeros(n ** 3, np.int64))
    H.itokmc_solve_field()
    assert rel_residual(H.itokmc_read_densities(itokmc.PHI), H.itokmc_read_densities(itokmc.RHO), ph) <= TOL
    H.close()


@pytest.mark.parametrize("guess", [0.0, 1e3, 1e18])
def test_noalloc_from_any_start_guess(guess):
    import torch
    ph = small_phys(64)
    rho = torch.from_numpy(charges("cloud", 64, 3) << 30).cuda()
    phi = torch.full((64 ** 3,), guess, dtype=torch.float64, device="cuda")
    E = torch.empty(3 * 64 ** 3, dtype=torch.float64, device="cuda")
    itokmc.itokmc_field_solve_noalloc(itokmc.make_config(ph, 1), rho, phi, E)
    assert rel_residual(phi.cpu().numpy(), rho.cpu().numpy(), ph) <= TOL


def test_no_charge_and_no_field():
    ph = small_phys(32, E0=0.0)
    H = itokmc.Handle(itokmc.make_config(ph, 100))
    H.itokmc_solve_field()
    assert not H.itokmc_read_densities(itokmc.PHI).any()
    H.close()
