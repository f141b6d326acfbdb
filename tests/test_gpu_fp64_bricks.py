"""The D3Q19 FP64 step and fields on their run-time bricks against the oracle: grids smaller than a brick,
ragged in every direction, with the body on a brick face or across a periodic edge, for every wall scheme.

One step from a common state.  Tolerance: about 290 operations of 1.1e-16 relative on values of the size
of f; 1e-13 times the largest |f| as in the other FP64 one-step tests.
"""
import numpy as np
import pytest

from oracle import lbm
from tests.harness import drop_on_cylinder

pytestmark = pytest.mark.gpu

GRIDS = [   # (nz, ny, nx), body, drop
    ((5, 6, 7), (3.0, 3.0, 2.0), 1.0, (3.0, 3.0, 3.5), 1.5),
    ((24, 24, 24), (12.0, 12.0, 9.0), 4.0, (12.0, 12.0, 18.0), 4.5),
    ((33, 17, 9), (4.0, 8.0, 16.0), 3.0, (4.0, 8.0, 24.0), 4.0),
    ((19, 40, 67), (66.0, 20.0, 9.0), 5.0, (66.0, 32.0, 9.0), 5.0),     # body across the periodic x edge
    ((2, 9, 35), (16.0, 4.0, 0.0), 1.0, (24.0, 4.0, 0.0), 3.0),         # two planes
]
WALLS = [dict(kappa=0.12), dict(kappa=-0.03), dict(wall="VD", rho_w_const=0.15), dict(wall="SF", Gw=-0.2),
         dict(eos_kind="PR", t_over_tc=0.86, sigma=0.11, kappa=0.1),
         dict(kappa=0.1, body_force=(2e-6, -1e-6, 3e-6), rates=dict(s_pi=1.3, s_m=1.6, s_nu=0.7))]


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("kw", WALLS)
def test_one_step_fp64_bricks(grid, kw):
    shape, c, R, dc, r = grid
    case = drop_on_cylinder(shape, c, R, dc, r, lattice="D3Q19", **kw)
    geo, p, _ = case.oracle()
    with case.gpu("fp64") as sim:
        sim.step(2)
        f0 = sim.get_state()
        _, rho, u = sim.observables(fields=True)
        sim.step(1)
        f1 = sim.get_state()
        assert sim.check_guards()[0] == 0
    ref = lbm.step(f0, geo, p)
    assert np.max(np.abs(f1 - ref)) < 1e-13 * max(1.0, np.abs(ref).max())
    _, rho_ref, u_ref = lbm.observables(f0, geo, p)
    fl = case.mask == 0
    assert np.max(np.abs(rho - rho_ref)[fl]) < 1e-13 * max(1.0, rho_ref.max())
    assert np.max(np.abs(u - u_ref)[:, fl]) < 1e-12      # divided by densities of 1e-2 and more
