"""The TMA z-march on grids of any width: the last columns moved inside the grid, rows padded to 16 bytes,
short pieces on small grids, and the fields pass on the same items.

One step from a common state against the oracle, with the FP32 one-step tolerance of the other march
tests (2e-6 of the largest |f|: the state carries 24-bit deviations, a step about 300 operations).  The
fields: the density is a sum of 19 stored values (4e-7 of the largest), u the ratio of sums of the same
size and a density of at least 1e-2.
"""
import numpy as np
import pytest

from oracle import lbm
from tests.harness import drop_on_cylinder

pytestmark = pytest.mark.gpu

GRIDS = {   # (nz, ny, nx), sphere centre (x, y, z), radius, drop centre, radius
    "97": ((21, 19, 97), (94.0, 9.0, 8.0), 4.0, (94.0, 9.0, 16.0), 5.0),     # 1 mod 4, body on the moved columns
    "66": ((12, 23, 66), (10.0, 20.0, 5.0), 3.0, (40.0, 20.0, 6.0), 5.0),    # 2 mod 4, body on the moved rows
    "43": ((33, 17, 43), (1.0, 1.0, 16.0), 4.0, (1.0, 1.0, 25.0), 5.0),      # 3 mod 4, body across two edges
    "40": ((4, 16, 40), (20.0, 8.0, 1.0), 1.5, (30.0, 8.0, 2.0), 4.0),       # the smallest grid the march takes
    "100": ((70, 24, 100), (50.0, 12.0, 30.0), 5.0, (50.0, 12.0, 41.0), 6.0),
    "39": ((9, 16, 39), (20.0, 8.0, 3.0), 2.0, (20.0, 8.0, 7.0), 3.0),       # below it: the z-pair march, padded rows
}


def _case(name, **kw):
    shape, c, R, dc, r = GRIDS[name]
    case = drop_on_cylinder(shape, c, R, dc, r, lattice="D3Q19", **kw)
    case.rho_ref = case.bounds()[0]
    return case


@pytest.mark.parametrize("name", sorted(GRIDS))
@pytest.mark.parametrize("kw", [dict(kappa=0.2), dict(wall="SF", Gw=-0.2, body_force=(2e-6, -1e-6, 3e-6)),
                                dict(wall="VD", rho_w_const=0.1)])
def test_step_and_fields(name, kw):
    case = _case(name, **kw)
    geo, p, _ = case.oracle()
    with case.gpu("fp32") as sim:
        assert sim.step_kernel() == ("pair" if name == "39" else "ztma")
        sim.step(3)
        s0 = sim.get_state()
        _, rho, u = sim.observables(fields=True)
        sim.step(1)
        s1 = sim.get_state()
        assert sim.check_guards() == (0, 0)
    ref = lbm.step(s0, geo, p)
    assert np.max(np.abs(s1 - ref)) <= 2e-6 * np.max(np.abs(ref))
    _, rho_ref, u_ref = lbm.observables(s0, geo, p)
    assert np.max(np.abs(rho - rho_ref)) <= 1e-6 * rho_ref.max()
    assert np.max(np.abs(u - u_ref)) <= 2e-5
    assert np.all(rho[case.mask != 0] == 0.0) and np.all(u[:, case.mask != 0] == 0.0)


@pytest.mark.parametrize("name", ["97", "66"])
def test_checkpoint_of_padded_rows(name):
    """A checkpoint holds 19 unpadded values per node and the step count, and reloads exactly."""
    from paper_1908_04443_gb300 import lbmwet as L
    case = _case(name, kappa=0.1)
    with case.gpu("fp32") as sim:
        sim.step(2)
        blob = L.lbm_save_state(sim.h)
        assert len(blob) == 19 * 4 * case.mask.size + 8
        sim.step(2)
        after = sim.get_state()
        L.lbm_load_state(sim.h, blob)
        sim.step(2)
        assert np.array_equal(sim.get_state(), after)
        assert sim.check_guards() == (0, 0)
