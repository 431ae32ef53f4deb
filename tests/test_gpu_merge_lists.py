"""Merge/split at the sizes and inputs where its kernels change over, bit for
bit against the oracle's merge of each cell's list: lists of 1 particle to
beyond the shared-memory tiers (chunks of 32, the tiers' capacities), 1 to 256
leaves, equal coordinates along one, two or all axes (which take the merge
that sorts per level), unit weights, and weights whose sum passes 2^31.  No
transport and no reactions (mu = D = 0, alpha = eta = 0), so the list of a
cell is what was set."""
import numpy as np
import pytest

import oracle
from gpu_util import gpu_handle, small_phys
from paper_2307_01797_gb300 import itokmc

pytestmark = pytest.mark.gpu

N = 8
SIZES = [1, 2, 3, 31, 32, 33, 63, 64, 65, 95, 96, 97, 128, 223, 224, 225, 300]


def cells_of(ph, kind, seed):
    rng = np.random.default_rng(seed)
    h = (ph["hi"][0] - ph["lo"][0]) / N
    out = []
    for k, m in enumerate(SIZES):
        c = 17 * k % (N ** 3)
        ijk = (c % N, (c // N) % N, c // (N * N))
        f = rng.uniform(0.01, 0.99, (3, m))
        if kind == "tie_one":
            f[k % 3] = rng.choice(f[k % 3], m)
        elif kind == "tie_two":
            f[k % 3], f[(k + 1) % 3] = 0.25, rng.choice([0.125, 0.5, 0.75], m)
        elif kind == "tie_all":
            f = f[:, rng.integers(0, max(1, m // 3), m)]
        w = rng.integers(1, 1000, m)
        if kind == "unit":
            w[:] = 1
        elif kind == "heavy":
            w = rng.integers(1, 2 ** 32 // (2 * m) + 2 ** 31 // m, m)
        X = np.stack([ph["lo"][a] + (ijk[a] + f[a]) * h for a in range(3)])
        out.append((c, X, w.astype(np.uint32)))
    return out


@pytest.mark.parametrize("ppc", [1, 2, 8, 32, 64, 128, 256])
@pytest.mark.parametrize("kind", ["distinct", "tie_one", "tie_two", "tie_all", "unit", "heavy"])
def test_merge_of_single_cells(kind, ppc):
    ph = small_phys(N, mu=0.0, D=0.0, alpha_A=0.0, eta=0.0, ppc=ppc, photon_ratio=0.0)
    lists = sorted(cells_of(ph, kind, seed=ppc), key=lambda q: q[0])
    X = np.concatenate([q[1] for q in lists], axis=1)
    w = np.concatenate([q[2] for q in lists])
    H = gpu_handle(ph, 4 * len(w) + 256 * len(lists))
    H.itokmc_set_particles(X[0], X[1], X[2], w)
    H.itokmc_set_field(*[np.zeros((N, N, N))] * 3)
    for stage in (itokmc.STAGE_TRANSPORT, itokmc.STAGE_KMC, itokmc.STAGE_PARTICLES):
        H.itokmc_run_stage(stage)
    G = H.itokmc_read_particles()
    at = 0
    for c, Y, wl in lists:
        x, y, z, wo = oracle.merge_list(Y[0], Y[1], Y[2], wl, ppc)
        sl = slice(at, at + len(wo))
        assert np.array_equal(G["w"][sl], wo) and np.array_equal(G["cell"][sl], np.full(len(wo), c))
        for k, v in (("x", x), ("y", y), ("z", z)):
            assert np.array_equal(G[k][sl].view(np.uint64), np.asarray(v).view(np.uint64)), (c, k)
        at += len(wo)
    assert at == len(G["w"])
    H.close()
