"""Merge/split of cells with copies of particles, in both forms: lists of up to
and beyond 32 elements in which copies stand together, apart, and beside
elements that are equal along one axis only.  Offsets are multiples of 1/64 of a
cell whose size is a power of two, so that both forms see the same coordinates,
extents and order: cells and weights are the oracle's, and so are the positions
(bit for bit in the FP64 form; in the mixed form to the rounding of a mean of at
most 96 FP32 terms, 96 * 2^-24 of a cell)."""
import numpy as np
import pytest

import oracle
from gpu_util import gpu_handle, small_phys
from paper_2307_01797_gb300 import itokmc

pytestmark = pytest.mark.gpu

N = 8
SIZES = [2, 3, 17, 31, 32, 33, 40, 64, 65, 95, 130, 200]


def lists(kind, seed):
    rng = np.random.default_rng(seed)
    for k, m in enumerate(SIZES):
        some = rng.permutation(64 ** 3)[:m]                      # distinct places
        f = np.stack([some % 64, some // 64 % 64, some // 4096]) / 64.0
        if kind == "together":
            f = np.repeat(f, 2, axis=1)[:, :m]
        elif kind == "apart":
            f = f[:, rng.integers(0, m // 2 + 1, m)]
        elif kind == "distinct":                                 # along every axis (m <= 64), else ties
            f = np.stack([rng.permutation(max(64, m))[:m] / max(64.0, m) for _ in range(3)])
            f = np.floor(f * 256) / 256
        yield 19 * k % N ** 3, f, rng.integers(1, 200, m).astype(np.uint32)


@pytest.mark.parametrize("ppc", [1, 4, 16, 32])
@pytest.mark.parametrize("kind", ["together", "apart", "one_axis", "distinct"])
@pytest.mark.parametrize("precision", [itokmc.FP64, itokmc.MIXED])
def test_copies(precision, kind, ppc):
    ph = small_phys(N, mu=0.0, D=0.0, alpha_A=0.0, eta=0.0, ppc=ppc, photon_ratio=0.0)
    ph["lo"], ph["hi"] = (0.0, 0.0, 0.0), (2.0 ** -7,) * 3
    h = 2.0 ** -10
    cells = sorted(lists(kind, ppc), key=lambda q: q[0])
    X = [np.concatenate([((c // N ** a) % N + f[a]) * h for c, f, _ in cells]) for a in range(3)]
    w = np.concatenate([q[2] for q in cells])
    H = gpu_handle(ph, 4 * len(w) + 256 * len(cells), precision=precision)
    H.itokmc_set_particles(*X, w)
    H.itokmc_set_field(*[np.zeros((N, N, N))] * 3)
    for stage in (itokmc.STAGE_TRANSPORT, itokmc.STAGE_KMC, itokmc.STAGE_PARTICLES):
        H.itokmc_run_stage(stage)
    G = H.itokmc_read_particles()
    at = 0
    for c, f, wl in cells:
        Y = [((c // N ** a) % N + f[a]) * h for a in range(3)]
        *pos, wo = oracle.merge_list(*Y, wl, ppc)
        sl = slice(at, at + len(wo))
        assert np.array_equal(G["w"][sl], wo) and (G["cell"][sl] == c).all()
        for k, v in zip("xyz", pos):
            if precision == itokmc.FP64:
                assert np.array_equal(G[k][sl].view(np.uint64), np.asarray(v).view(np.uint64)), (c, k)
            else:
                assert np.abs(G[k][sl] - v).max() <= 96 * 2.0 ** -24 * h, (c, k)
        at += len(wo)
    assert at == len(G["w"])
    H.close()
