"""FP64 Poisson draws on the device (their floors and comparisons are decided
in pairs of floats and, near a boundary, in FP64) against the oracle's, at the
means where a branch begins or ends.  Counts are whole numbers: no tolerance."""
import numpy as np
import pytest

import oracle
from paper_2307_01797_gb300 import itokmc, synth

from gpu_util import assert_particles_equal, gpu_handle, small_phys

pytestmark = pytest.mark.gpu


# tiny means, the search's end at 10, ordinary means, the pairs' end at 2^24
# (the density falls by a third over the grid: 1.2 * 2^24 has both sides), and
# far above it
@pytest.mark.parametrize("mu", [1e-25, 1e-3, 0.7, 9.999, 12.0, 60.0, 4096.5, 1e6, 1.2 * 2.0 ** 24, 3e9])
def test_seeded_counts_equal_the_oracle(mu):
    n = 32
    ph = small_phys(n)
    h = synth.cell_size(ph)
    L = n * h
    blobs = [dict(center=(0.3 * L, 0.5 * L, 0.6 * L), sigma=1.1 * L, peak=mu / h ** 3)]
    st, counts = oracle.seed_blobs(oracle.make_params(ph, seed=77), blobs)
    H = gpu_handle(ph, n ** 3 * ph["ppc"], seed0=77)
    H.itokmc_seed_blobs(blobs, itokmc.SEED_NEUTRAL)
    assert np.array_equal(H.itokmc_read_densities(itokmc.NPOS), counts)
    assert_particles_equal(H.itokmc_read_particles(), st)
    H.close()


@pytest.mark.parametrize("eps", [0.03, float("inf")])
def test_short_and_long_waiting_times_equal_the_oracle(eps):
    """Exponential times are compared in FP32 first: cells whose total rate
    times dt lies around one, with critical reactions (few electrons, strong
    attachment)."""
    ph = dict(small_phys(8), eps=eps, eta=4e5)
    for E, X0, dt in ((1e6, 3, 2e-11), (2e6, 1, 5e-11), (3e6, 6, 1e-11), (3e6, 20, 4e-12)):
        ph["dt"] = dt
        ref = oracle.kmc0d(oracle.make_params(ph, seed=5), E, X0, 2000, 30)
        got = itokmc.itokmc_kmc0d(itokmc.make_config(ph, 1, seed0=5), E, X0, 2000, 30)
        assert np.array_equal(got, ref)
