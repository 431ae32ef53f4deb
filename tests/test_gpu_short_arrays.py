"""Device arrays that end before the count that the call states are refused, as
the copies of them were, before any kernel reads them; the handle stays usable.
Arrays that end exactly there, and arrays inside a larger allocation, are taken."""
import ctypes

import numpy as np
import pytest

from gpu_util import gpu_handle, small_phys
from paper_2307_01797_gb300 import itokmc

pytestmark = pytest.mark.gpu

N = 1 << 20


@pytest.fixture
def memory():
    """cudaMalloc of the runtime that torch has loaded."""
    import torch
    torch.zeros(1, device="cuda")
    rt = ctypes.CDLL("libcudart.so.13")
    rt.cudaMalloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
    rt.cudaFree.argtypes = [ctypes.c_void_p]
    rt.cudaMemset.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t]
    got = []

    def alloc(nbytes):
        p = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(p), nbytes) == 0
        assert rt.cudaMemset(p, 0, nbytes) == 0
        got.append(p)
        return p
    yield alloc
    for p in got:
        rt.cudaFree(p)


@pytest.mark.parametrize("precision", [itokmc.FP64, itokmc.MIXED])
@pytest.mark.parametrize("short", range(5))
def test_short_particle_arrays(memory, short, precision):
    import torch
    ph = small_phys(8)
    H = gpu_handle(ph, N, precision=precision)
    h = (ph["hi"][0] - ph["lo"][0]) / 8
    # a particle in the first cell each: all bytes of x, y and z are in the domain
    x = torch.full((N,), ph["lo"][0] + 0.5 * h, dtype=torch.float64, device="cuda")
    w = torch.ones(N, dtype=torch.int32, device="cuda")
    r = torch.zeros(N, dtype=torch.int32, device="cuda")
    args = [ctypes.c_void_p(t.data_ptr()) for t in (x, x, x, w, r)]
    full = list(args)
    args[short] = memory(4096)
    L = itokmc.lib()
    assert L.itokmc_set_particles(H.h, *args, N, itokmc.DEVICE) == -1      # ERR_ARG
    assert b"fewer" in L.itokmc_last_error(H.h)
    # arrays that end where they should: 1024 realizations' indices of zero
    m = 4096 // (8 if short < 3 else 4)
    if short == 4:
        assert L.itokmc_set_particles(H.h, *full[:4], args[4], m, itokmc.DEVICE) == 0
        assert H.itokmc_num_particles() == m
    assert L.itokmc_set_particles(H.h, *full, N, itokmc.DEVICE) == 0
    P = H.itokmc_read_particles()
    assert len(P["w"]) == N and (P["w"] == 1).all() and np.allclose(P["x"], ph["lo"][0] + 0.5 * h)
    H.close()


def test_short_field(memory):
    import torch
    ph = small_phys(16)
    H = gpu_handle(ph, 100)
    p = memory(3 * 16 ** 3 * 8 - 8)
    L = itokmc.lib()
    assert L.itokmc_set_field(H.h, p, itokmc.DEVICE) == -1
    assert b"fewer" in L.itokmc_last_error(H.h)
    # exactly as long, and inside a larger allocation up to its end
    q = memory(3 * 16 ** 3 * 8 + 8)
    for o in (0, 8):
        assert L.itokmc_set_field(H.h, ctypes.c_void_p(q.value + o), itokmc.DEVICE) == 0
    assert not H.itokmc_read_densities(itokmc.E).any()
    H.close()
