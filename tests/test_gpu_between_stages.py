"""Calls that the stage order admits between two stages and that use the device
counters themselves: the field of the current charge after the chemistry (which
is the last to read the field), and the autotuner after the transport or the
chemistry.  The stages then end as without the call: the attached electrons are
removed, the photons are emitted, the totals are the same, all to the last bit."""
import numpy as np
import pytest

from paper_2307_01797_gb300 import itokmc, synth

from gpu_util import assert_particles_equal, gpu_handle, mixed_state, small_phys

pytestmark = pytest.mark.gpu

TOTALS = ("ionizations", "attachments", "photon_emissions", "photons_absorbed_weight", "photons_lost_weight",
          "n_new_particles", "merge_cells", "merge_elements")


def run(ph, st, precision, call, after):
    E = synth.random_field(ph, seed=4, amp=5e5, base=4.5e6)
    H = gpu_handle(ph, 16 * len(st["w"]) + 200000, seed0=9, precision=precision)
    H.itokmc_set_particles(st["x"], st["y"], st["z"], st["w"])
    H.itokmc_set_field(*E)
    for stage in (itokmc.STAGE_TRANSPORT, itokmc.STAGE_KMC, itokmc.STAGE_PARTICLES):
        H.itokmc_run_stage(stage)
        if call and stage == after:
            getattr(H, call)()
    out = H.itokmc_read_particles(), H.itokmc_read_densities(itokmc.NPOS), H.itokmc_get_stats()
    H.close()
    return out


@pytest.mark.parametrize("precision", [itokmc.FP64, itokmc.MIXED])
@pytest.mark.parametrize("call,after", [("itokmc_solve_field", itokmc.STAGE_KMC), ("itokmc_autotune", itokmc.STAGE_KMC),
                                        ("itokmc_autotune", itokmc.STAGE_TRANSPORT)])
@pytest.mark.parametrize("what", ["attachment", "photons"])
def test_stages_end_as_without_the_call(what, call, after, precision):
    ph = small_phys(16, dt=5e-11, photon_ratio=1.0 if what == "photons" else 0.0)
    if what == "attachment":
        ph.update(alpha_A=0.0, eta=0.3 / (ph["dt"] * ph["mu"] * 4.5e6))
    st = mixed_state(ph, seed=11, n_random=2000, peak=2e18)
    want, got = run(ph, st, precision, None, None), run(ph, st, precision, call, after)
    assert want[2]["attachments"] > 0.05 * st["w"].sum() if what == "attachment" else want[2]["photons_absorbed_weight"] > 0
    assert_particles_equal(got[0], want[0])
    assert np.array_equal(got[1], want[1])
    assert [got[2][k] for k in TOTALS] == [want[2][k] for k in TOTALS]
