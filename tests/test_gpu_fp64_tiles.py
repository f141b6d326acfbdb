"""The D2Q9 FP64 step on its run-time tiles against the oracle: grids whose tiles are ragged, narrower
than a tile, one node high, or cut small for a small grid, with the body on a tile edge or across the
periodic edge, for every wall scheme and equation of state.

One step from a common state.  Tolerance: a step is about 140 operations on values of the size of f, each
rounded at 1.1e-16 relative; 1e-13 times the largest |f| is two orders above their sum (the bound of the
other FP64 one-step tests).
"""
import numpy as np
import pytest

from oracle import lbm
from tests.harness import drop_on_cylinder

pytestmark = pytest.mark.gpu

GRIDS = [
    ((100, 100), (50.0, 30.0), 15.0, (50.0, 62.0), 18.0),      # about one tile per SM
    ((5, 7), (3.0, 2.0), 1.0, (3.0, 3.5), 1.5),                # smaller than a tile and its halo
    ((3, 130), (60.0, 1.0), 0.5, (20.0, 1.0), 3.0),            # three rows
    ((17, 41), (40.0, 8.0), 5.0, (20.0, 8.0), 5.0),            # body across the periodic x edge, ragged
    ((259, 321), (64.0, 130.0), 33.0, (64.0, 190.0), 30.0),    # large tiles, ragged by one node
]
WALLS = [dict(kappa=0.12), dict(kappa=-0.03), dict(wall="VD", rho_w_const=0.15), dict(wall="SF", Gw=-0.2),
         dict(eos_kind="PR", t_over_tc=0.86, sigma=0.11, kappa=0.1),
         dict(kappa=0.1, body_force=(2e-6, -1e-6, 0.0))]


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("kw", WALLS)
def test_one_step_fp64_tiles(grid, kw):
    shape, c, R, dc, r = grid
    case = drop_on_cylinder(shape, c, R, dc, r, **kw)
    geo, p, _ = case.oracle()
    with case.gpu("fp64") as sim:
        sim.step(2)
        f0 = sim.get_state()
        _, rho, u = sim.observables(fields=True)
        sim.step(1)
        f1 = sim.get_state()
    ref = lbm.step(f0, geo, p)
    assert np.max(np.abs(f1 - ref)) < 1e-13 * max(1.0, np.abs(ref).max())
    _, rho_ref, u_ref = lbm.observables(f0, geo, p)
    fl = case.mask == 0
    assert np.max(np.abs(rho - rho_ref)[fl]) < 1e-13 * max(1.0, rho_ref.max())
    assert np.max(np.abs(u - u_ref)[:, fl]) < 1e-12      # divided by densities of 1e-2 and more
