"""lbm_step_kernel_used names the D3Q19 FP32 kernel that runs: the TMA-staged z-march from 40 x 16 x 4 nodes on,
the z-pair march below, whatever the width and whether the march was asked for or not.  On the grids below the
limit the state equals that of the z-pair march asked for by name, bit for bit.
"""
import numpy as np
import pytest

from tests.harness import drop_on_cylinder

pytestmark = pytest.mark.gpu

# (nz, ny, nx)
SMALL = [(9, 16, 36), (9, 12, 64), (3, 16, 64), (12, 20, 16)]     # widths that are multiples of 4
LARGE = [(4, 16, 40), (9, 17, 41)]


def _case(shape, kernel):
    nz, ny, nx = shape
    return drop_on_cylinder(shape, (nx / 2, ny / 2, 1.0), 1.5, (nx / 2, ny / 2, nz / 2), 3.0, lattice="D3Q19",
                            kappa=0.1, step_kernel=kernel)


def _run(shape, kernel):
    with _case(shape, kernel).gpu("fp32") as sim:
        name = sim.step_kernel()
        sim.step(3)
        return name, sim.get_state()


@pytest.mark.parametrize("kernel", ["auto", "ztma"])
@pytest.mark.parametrize("shape", SMALL)
def test_small_grids_report_the_z_pair_march(shape, kernel):
    name, f = _run(shape, kernel)
    assert name == "pair"
    assert np.array_equal(f, _run(shape, "pair")[1])


@pytest.mark.parametrize("shape", LARGE)
def test_grids_of_the_march_report_it(shape):
    assert _run(shape, "auto")[0] == "ztma"
    assert _run(shape, "pair")[0] == "pair"
