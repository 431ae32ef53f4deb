"""Electrons lost and photons emitted, where their kernels change course: cells
with one particle, with more than four and not a multiple of four, with weights
whose products need 32 bits, 64 or more; few and many photon-emitting cells,
with up to n_new samples each.  Everything against the oracle, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2307_01797_gb300 import itokmc, synth

from gpu_util import assert_particles_equal, gpu_handle, oracle_state, small_phys

pytestmark = pytest.mark.gpu


def check(ph, st, seed):
    E = synth.random_field(ph, seed=seed, amp=5e5, base=4.5e6)
    n3 = ph["n"] ** 3
    S = oracle_state(ph, st, seed, np.zeros(n3, np.int64), np.zeros(n3, np.int64))
    new, info = oracle.step(oracle.make_params(ph, seed=seed, step=0), S, E)
    H = gpu_handle(ph, 4 * len(st["w"]) + 64 * n3, seed0=seed)
    H.itokmc_set_particles(st["x"], st["y"], st["z"], st["w"])
    H.itokmc_set_field(*E)
    for stage in (itokmc.STAGE_TRANSPORT, itokmc.STAGE_KMC, itokmc.STAGE_PARTICLES):
        H.itokmc_run_stage(stage)
    assert_particles_equal(H.itokmc_read_particles(), new)
    assert np.array_equal(H.itokmc_read_densities(itokmc.NPOS), new["Npos"])
    H.close()
    return info


@pytest.mark.parametrize("wmax,per", [(1, 1), (3, 7), (40000, 9), (10 ** 6, 33), (4 * 10 ** 9, 2), (4 * 10 ** 9, 6)])
def test_losses_by_attachment(wmax, per):
    # attachment alone: alpha = 0, a tenth to a half of the electrons lost; eight
    # fraction bits, so that 2.4e10 electrons in a cell fit the fixed-point density
    ph = small_phys(8, alpha_A=0.0, eta=2e4, dt=2e-10, ppc=64, D=0.0, mu=1e-4, frac_bits=8)
    ph["eta"] = 0.3 / (ph["dt"] * ph["mu"] * 4.5e6)
    rng = np.random.default_rng(per)
    L, h = ph["hi"][0], ph["hi"][0] / 8
    cells = rng.choice(8 ** 3, 60, replace=False)
    c = np.repeat(cells, per)
    pos = (np.stack([c % 8, c // 8 % 8, c // 64]) + rng.uniform(0.2, 0.8, (3, len(c)))) * h
    st = dict(x=pos[0], y=pos[1], z=pos[2], w=rng.integers((wmax + 1) // 2, wmax + 1, len(c)).astype(np.uint32))
    info = check(ph, st, 40 + per)
    assert info["n_att"].sum() > 0.05 * st["w"].sum(dtype=np.float64) and info["n_ion"].sum() == 0


@pytest.mark.parametrize("n,count,wmax,ratio", [(8, 3, 1, 1.0), (8, 200, 10 ** 5, 0.5), (16, 60000, 100, 2.0), (32, 120000, 30, 1.0)])
def test_photons_of_few_and_many_cells(n, count, wmax, ratio):
    ph = small_phys(n, photon_ratio=ratio, dt=2e-11)
    st = synth.random_particles(ph, count, seed=n, wmax=wmax, margin=0.02)
    info = check(ph, st, 60 + n)
    assert count < 10 or info["n_ph"].sum() > 30
