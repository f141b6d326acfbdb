"""Kernels that are set up while the one before them ends: a sequence of calls issued without a pause gives,
bit for bit, what it gives with a device synchronisation after every call (every dependence between two
launches is on the whole of the earlier one).  Each kernel family, on grids of a few CTAs and of many.
"""
import numpy as np
import pytest

from tests.harness import drop_on_cylinder

pytestmark = pytest.mark.gpu

GRIDS = [   # shape, body, drop, lattice, precision
    ((40, 48), (24.0, 14.0), 6.0, (24.0, 28.0), 7.0, "D2Q9", "fp32"),
    ((350, 301), (150.0, 130.0), 50.0, (150.0, 240.0), 60.0, "D2Q9", "fp32"),
    ((40, 48), (24.0, 14.0), 6.0, (24.0, 28.0), 7.0, "D2Q9", "fp64"),
    ((150, 131), (65.0, 50.0), 20.0, (65.0, 95.0), 24.0, "D2Q9", "fp64"),
    ((40, 41, 44), (22.0, 20.0, 14.0), 6.0, (22.0, 20.0, 28.0), 7.0, "D3Q19", "fp32"),
    ((24, 25, 26), (13.0, 12.0, 9.0), 4.0, (13.0, 12.0, 18.0), 4.5, "D3Q19", "fp64"),
]


def sequence(case, precision, sync):
    import torch
    out = []
    with case.gpu(precision) as sim:
        rho = torch.zeros(case.mask.size, dtype=torch.float64, device="cuda")
        u = torch.zeros(case.mask.ndim * case.mask.size, dtype=torch.float64, device="cuda")
        if not sync:
            torch.cuda.synchronize()

        def call(f, *a):
            f(*a)
            if sync:
                torch.cuda.synchronize()

        from paper_1908_04443_gb300 import lbmwet as L
        for n in (1, 1, 1, 16, 2, 33, 1):
            call(sim.enqueue, n)
            call(L.lbm_fields_device, sim.h, rho.data_ptr(), u.data_ptr())
            call(L.lbm_fields_device, sim.h, rho.data_ptr(), u.data_ptr())
        sim.step(1)
        torch.cuda.synchronize()
        out += [rho.cpu().numpy(), u.cpu().numpy(), sim.get_state()]
        assert sim.check_guards()[0] == 0
    return out


@pytest.mark.parametrize("grid", GRIDS)
def test_calls_in_a_row_as_one_by_one(grid):
    shape, c, R, dc, r, lattice, precision = grid
    case = drop_on_cylinder(shape, c, R, dc, r, lattice=lattice, kappa=0.08)
    for a, b in zip(sequence(case, precision, False), sequence(case, precision, True)):
        assert np.array_equal(a, b)
