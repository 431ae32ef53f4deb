"""Device memory that a handle takes through its caller's allocator, in bytes: no
more than the budgets that sufficed when the solve ran on FP64 arrays and the
merge sorted per level."""
import pytest

from gpu_util import small_phys
from paper_2307_01797_gb300 import itokmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,precision,field_precision,mobile,capacity,budget", [
    (64, 1, 0, -1, 0, 300000, 210860288),
    (64, 1, 1, -1, 0, 300000, 195271936),
    (64, 1, 1, 0, 0, 300000, 195271936),
    (64, 1, 0, 1, 0, 300000, 210860288),
    (64, 1, 0, -1, 1, 300000, 256997632),
    (8, 16, 0, -1, 0, 1000, 106088960),
    (8, 16, 1, -1, 0, 1000, 105803264),
    (32, 3, 0, -1, 0, 1000, 132719104),
    (32, 3, 1, -1, 0, 1000, 129549824),
    (128, 1, 0, -1, 0, 1000, 723401984),
    (128, 1, 1, -1, 0, 1000, 656269568),
    (32, 16, 0, -1, 1, 300000, 380592896),
])
def test_a_budget_that_sufficed(monkeypatch, n, R, precision, field_precision, mobile, capacity, budget):
    taken = []
    alloc = itokmc._TorchAllocator._alloc

    def counted(self, nbytes, ctx):
        if sum(taken) + nbytes > budget:
            return None
        taken.append(nbytes)
        return alloc(self, nbytes, ctx)
    monkeypatch.setattr(itokmc._TorchAllocator, "_alloc", counted)
    ph = small_phys(n)
    if mobile:
        ph.update(mobile_ions=True, mu_ion=2e-4, D_ion=1e-6)
    H = itokmc.Handle(itokmc.make_config(ph, capacity, realizations=R, precision=precision, field_precision=field_precision))
    H.itokmc_solve_field()
    H.close()
