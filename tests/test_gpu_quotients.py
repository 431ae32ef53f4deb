"""The FP64 push's grid quotients at the points where their rounding decides
something: cell faces and centres and up to four ulps beside them, the walls
and their half cells, on grids whose cell size is or is not a short binary
fraction and whose corner is or is not the origin.  Bit for bit against the
oracle: with E = 0 and D = 0 the particles stay where they are and the cell,
the stencil and the fixed-point deposit come from those points; with a field
the interpolation weights do (D = 0: no draw moves the points)."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_particles_equal, gpu_handle, oracle_state, small_phys
from paper_2307_01797_gb300 import itokmc, synth

pytestmark = pytest.mark.gpu

# corner, edge length, cells per axis
GRIDS = [(0.0, 0.01, 16), (0.0, 1.0 / 64, 8), (-0.0031, 0.0069, 16), (0.7, 0.713, 32), (0.0, 0.02, 64), (-2.0, 1.0, 8)]


def edge_points(lo, hi, n, count, rng):
    h = (hi - lo) / n
    base = lo + np.concatenate([np.arange(n), np.arange(n) + 0.5, rng.random(2 * n) * n]) * h
    pts = []
    for k in range(-4, 5):
        p = base.copy()
        for _ in range(abs(k)):
            p = np.nextafter(p, np.inf if k > 0 else -np.inf)
        pts.append(p)
    pts = np.concatenate(pts + [[lo, np.nextafter(hi, -np.inf)]])
    pts = pts[(pts >= lo) & (pts < hi)]
    return rng.choice(pts, (3, count))


@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("lo,hi,n", GRIDS)
def test_push_at_faces_and_centres(lo, hi, n, field):
    rng = np.random.default_rng(n + int(1e4 * hi))
    ph = small_phys(n, lo=(lo,) * 3, hi=(hi,) * 3, D=0.0, dt=1e-13)
    X = edge_points(lo, hi, n, 6000, rng)
    st = dict(x=X[0], y=X[1], z=X[2], w=rng.integers(1, 1 << 20, X.shape[1]).astype(np.uint32))
    E = synth.random_field(ph, seed=3, amp=3e6) if field else tuple(np.zeros((n, n, n)) for _ in range(3))
    H = gpu_handle(ph, 2 * len(st["w"]) + 1000)
    H.itokmc_set_particles(st["x"], st["y"], st["z"], st["w"])
    H.itokmc_set_field(*E)
    H.itokmc_run_stage(itokmc.STAGE_TRANSPORT)
    S = oracle_state(ph, st, 1)
    p = oracle.make_params(ph, seed=1, step=0)
    xo, yo, zo, cell = oracle.push(p, S["x"], S["y"], S["z"], E)
    perm = oracle.sort_by_cell(cell, n ** 3)
    T = dict(x=xo[perm], y=yo[perm], z=zo[perm], w=S["w"][perm], cell=cell[perm])
    assert_particles_equal(H.itokmc_read_particles(), T)
    ne, Xe = oracle.deposit(p, T["x"], T["y"], T["z"], T["w"], T["cell"])
    assert np.array_equal(H.itokmc_read_densities(itokmc.NE_FIX), ne)
    assert np.array_equal(H.itokmc_read_densities(itokmc.XE), Xe)
    # the deposit alone (an initial field) gives the same densities
    H.itokmc_solve_field()
    assert np.array_equal(H.itokmc_read_densities(itokmc.NE_FIX), ne)
    H.close()
