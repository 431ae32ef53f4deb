"""Particle upload: the same particles from host memory, from device memory,
from device memory at an odd address, in cell order (where the sort is skipped)
and one swap away from it give the same canonical list, bit for bit (both
forms, one realization and three, ion species)."""
import ctypes

import numpy as np
import pytest

from gpu_util import small_phys
from paper_2307_01797_gb300 import itokmc, synth

pytestmark = pytest.mark.gpu


def canonical_order(ph, P, real, species, R):
    n = ph["n"]
    h = (ph["hi"][0] - ph["lo"][0]) / n
    c = [np.clip(np.floor((P[k] - ph["lo"][a]) / h).astype(np.int64), 0, n - 1) for a, k in enumerate("xyz")]
    cell = (c[2] * n + c[1]) * n + c[0]
    return np.argsort((species * R + real) * n ** 3 + cell, kind="stable")


@pytest.mark.parametrize("precision", [itokmc.FP64, itokmc.MIXED])
@pytest.mark.parametrize("R,mobile", [(1, False), (3, False), (2, True)])
def test_upload_paths_agree(precision, R, mobile):
    import torch
    ph = small_phys(16)
    if mobile:
        ph = synth.with_mobile_ions(ph)
        ph["mobile_ions"] = True
    rng = np.random.default_rng(R)
    P = synth.random_particles(ph, 20011, seed=4)
    real = rng.integers(0, R, 20011).astype(np.int32)
    species = rng.integers(0, 3 if mobile else 1, 20011).astype(np.int32)

    def upload(order, how):
        a = [np.ascontiguousarray(P[k][order]) for k in "xyz"] + [P["w"][order], real[order], species[order]]
        H = itokmc.Handle(itokmc.make_config(ph, 40000, realizations=R, precision=precision))
        if how == "host":
            H.itokmc_set_particles_species(*a[:4], a[5], realization=a[4])
        else:
            shift = 4 if how == "odd" else 0
            keep, ptr = [], []
            for v in a:
                t = torch.empty(v.nbytes + 64, dtype=torch.uint8, device="cuda")
                t[shift:shift + v.nbytes] = torch.from_numpy(v.view(np.uint8)).cuda()
                keep.append(t)
                ptr.append(ctypes.c_void_p(t.data_ptr() + shift))
            code = itokmc.lib().itokmc_set_particles_species(H.h, ptr[0], ptr[1], ptr[2], ptr[3], ptr[4], ptr[5], len(a[3]),
                                                             itokmc.DEVICE)
            assert code == 0, itokmc.lib().itokmc_last_error(H.h)
        out = H.itokmc_read_particles()
        H.close()
        return out

    mixed_order = np.arange(20011)
    want = upload(mixed_order, "host")
    sorted_order = canonical_order(ph, P, real, species, R)
    swapped = sorted_order.copy()
    swapped[[10, 15000]] = swapped[[15000, 10]]
    for order, how in ((mixed_order, "device"), (mixed_order, "odd"), (sorted_order, "host"), (sorted_order, "device")):
        got = upload(order, how)
        for k in want:
            assert np.array_equal(got[k], want[k]), (how, k)
    got = upload(swapped, "device")
    assert np.array_equal(np.sort(got["w"]), np.sort(want["w"])) and np.array_equal(got["cell"], want["cell"])


def test_fp32_field_takes_the_same_modulus():
    """The mixed form's |E| of an FP32-valued field against the FP64 formula,
    through the KMC: cells of one electron count under fields whose components
    are FP32 numbers fire as under the same field a part in 2^40 away (no FP32
    number, so |E| goes through FP64, and rounds to the same FP32 value)."""
    ph = small_phys(16, dt=5e-12, alpha_B=1e7)
    E = [np.float32(v).astype(np.float64) for v in synth.random_field(ph, seed=9, amp=8e6)]
    st = synth.random_particles(ph, 30000, seed=2)
    fired = []
    for f in (1.0, 1.0 + 2.0 ** -40):
        H = itokmc.Handle(itokmc.make_config(ph, 100000, precision=itokmc.MIXED))
        H.itokmc_set_particles(st["x"], st["y"], st["z"], st["w"])
        H.itokmc_set_field(*[v * f for v in E])
        H.itokmc_run_stage(itokmc.STAGE_TRANSPORT)
        H.itokmc_run_stage(itokmc.STAGE_KMC)
        fired.append(H.itokmc_read_densities(itokmc.FIRINGS))
        H.close()
    assert fired[0].sum() > 10000
    assert np.array_equal(fired[0], fired[1])
