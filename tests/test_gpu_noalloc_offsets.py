"""The allocation-free field solve with caller arrays at any offset that the ABI
admits (a multiple of 8 bytes): the same potential and field, bit for bit, as
with arrays at 16-byte boundaries, also where the start guess lies beyond the
integers' range (FP64 cycles, which load and store pairs of values)."""
import numpy as np
import pytest

from gpu_util import small_phys
from paper_2307_01797_gb300 import itokmc
from test_gpu_field_forms import charges

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("guess", [0.0, 1e18])
@pytest.mark.parametrize("precision", [itokmc.FP64, itokmc.MIXED])
@pytest.mark.parametrize("n", [8, 32, 64])
def test_arrays_at_odd_offsets(n, precision, guess):
    import torch
    ph = small_phys(n)
    n3 = n ** 3
    out = []
    for o in (0, 1):
        rho = torch.zeros(n3 + 2, dtype=torch.int64, device="cuda")
        phi = torch.full((n3 + 2,), -7.0, dtype=torch.float64, device="cuda")
        E = torch.full((3 * n3 + 2,), -7.0, dtype=torch.float64, device="cuda")
        assert phi.data_ptr() % 16 == 0
        rho[o:o + n3] = torch.from_numpy(charges("cloud", n, 3) << 30).cuda()
        phi[o:o + n3] = guess
        res = itokmc.itokmc_field_solve_noalloc(itokmc.make_config(ph, 1, precision=precision), rho[o:o + n3],
                                                phi[o:o + n3], E[o:o + 3 * n3])
        out.append((res, phi[o:o + n3].cpu().numpy(), E[o:o + 3 * n3].cpu().numpy()))
        # nothing beside the arrays
        assert (torch.cat([phi[:o], phi[o + n3:], E[:o], E[o + 3 * n3:]]) == -7.0).all()
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][2], out[1][2])
