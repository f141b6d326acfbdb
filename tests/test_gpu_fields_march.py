"""The fields pass of the TMA-staged z-march (FP32) gives, bit for bit, what the scalar z-march's gives for the same
state: both round density, psi, force and velocity alike, so the fields are no further from 64 bits on the grids
that the march takes than on the others.  Widths of every remainder, items with and without solids, every wall scheme.
"""
import numpy as np
import pytest

from tests.harness import drop_on_cylinder

pytestmark = pytest.mark.gpu

GRIDS = [   # (nz, ny, nx), sphere centre (x, y, z), radius, drop centre, radius
    ((40, 24, 96), (48.0, 12.0, 14.0), 4.0, (48.0, 12.0, 24.0), 6.0),
    ((21, 19, 97), (94.0, 9.0, 8.0), 4.0, (94.0, 9.0, 16.0), 5.0),
    ((33, 17, 43), (1.0, 1.0, 16.0), 4.0, (1.0, 1.0, 25.0), 5.0),
]


@pytest.mark.parametrize("grid", range(len(GRIDS)))
@pytest.mark.parametrize("kw", [dict(kappa=0.2), dict(kappa=-0.03, body_force=(2e-6, -1e-6, 3e-6)),
                                dict(wall="SF", Gw=-0.2), dict(wall="SF", Gw=-0.2, body_force=(2e-6, -1e-6, 3e-6)),
                                dict(wall="VD", rho_w_const=0.1),
                                dict(eos_kind="PR", t_over_tc=0.86, kappa=0.1)])
def test_fields_of_one_state_by_both_marches(grid, kw):
    from paper_1908_04443_gb300 import lbmwet as L
    out = []
    blob = None
    for kernel in ("ztma", "tile"):
        case = drop_on_cylinder(*GRIDS[grid], lattice="D3Q19", **kw)
        case.rho_ref = case.bounds()[0]
        case.step_kernel = kernel
        with case.gpu("fp32") as sim:
            if blob is None:
                sim.step(20)
                blob = L.lbm_save_state(sim.h)
            else:
                L.lbm_load_state(sim.h, blob)
            assert sim.step_kernel() == kernel
            out.append(sim.observables(fields=True)[1:])
    (rho_a, u_a), (rho_b, u_b) = out
    assert np.array_equal(rho_a, rho_b)
    assert np.array_equal(u_a, u_b)
