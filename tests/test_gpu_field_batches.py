"""Large FP32 grids interpolate the coarse correction plane by plane up the
grid, smaller ones cell group by cell group, with the same operations: a batch
of two equal 256^3 realizations (2^25 cells) has the potential of one alone,
bit for bit."""
import numpy as np
import pytest

from paper_2307_01797_gb300 import itokmc

from gpu_util import small_phys

pytestmark = pytest.mark.gpu


def test_a_batch_has_the_potential_of_one_alone():
    n = 256
    ph = small_phys(n)
    rng = np.random.default_rng(9)
    pos = np.zeros(n ** 3, np.int64)
    # a cloud, and charges at the electrodes and the corners
    pos[rng.integers(0, n ** 3, 20000)] = 1000
    pos[[0, n - 1, n ** 3 - 1, n ** 3 - n]] = 50000
    phi = []
    for R in (1, 2):
        H = itokmc.Handle(itokmc.make_config(ph, 100, realizations=R, precision=itokmc.MIXED))
        H.itokmc_set_ions(np.tile(pos, R), np.zeros(R * n ** 3, np.int64))
        H.itokmc_solve_field()
        phi.append(H.itokmc_read_densities(itokmc.PHI, -1).reshape(R, -1))
        H.close()
    assert np.array_equal(phi[1][0], phi[0][0]) and np.array_equal(phi[1][1], phi[0][0])
