"""The adjoint on grids its 32 x 8 tiles do not fit: narrower than a tile and its halo, ragged in both
directions, the body across a periodic edge; and with buffers too large for the memory pool.

Tolerance: as for the other FP64 gradients against central differences of the oracle (1e-6 of the largest
derivative: the differences' own error at a step of 1e-5); equal bits where only the buffers differ.  FP32
against FP64 for one loss, linear in the final density: 2e-3 of the largest derivative, as for the other FP32
gradients (single-precision rounding of states and adjoints over more steps than here).
"""
import numpy as np
import pytest

from oracle import gradient as GR
from tests.harness import drop_on_cylinder

pytestmark = pytest.mark.gpu

N_STEPS = 9
GRIDS = [   # (ny, nx), body, drop
    ((13, 12), (6.0, 4.0), 2.3, (6.0, 9.0), 2.5),
    ((17, 33), (0.0, 8.0), 3.2, (8.0, 8.0), 4.0),      # body across the periodic x edge, one node over a tile
    ((9, 70), (34.0, 0.0), 2.4, (41.0, 4.0), 3.5),     # across y, where the last tile of a column is one row
    ((35, 37), (31.0, 9.0), 5.0, (31.0, 20.0), 6.0),   # across a tile corner
]


def gradient(case, kappa, target, every):
    import torch
    from paper_1908_04443_gb300 import lbmwet as L
    case.kappa = kappa
    with case.gpu("fp64", stream=torch.cuda.current_stream()) as sim:
        L.lbm_record(sim.h, N_STEPS, every)
        rho = torch.zeros(sim.n, dtype=torch.float64, device="cuda")
        L.lbm_fields_device(sim.h, rho.data_ptr(), None)
        fluid = torch.as_tensor((case.mask.reshape(-1) == 0), device="cuda")
        tgt = torch.as_tensor(target.reshape(-1), device="cuda")
        drho = torch.where(fluid, 2.0 * (rho - tgt), torch.zeros_like(rho))
        return L.lbm_adjoint(sim.h, drho.data_ptr(), len(kappa))


def problem(grid):
    shape, c, R, dc, r = grid
    case = drop_on_cylinder(shape, c, R, dc, r, kappa=0.1)
    geo, p, f0 = case.oracle()
    nw = len(geo.wall_flat)
    rng = np.random.default_rng(5)
    kappa = rng.uniform(0.02, 0.3, nw)
    _, target = GR.loss(f0, geo, p, kappa + 0.08 * rng.uniform(-1, 1, nw), N_STEPS, np.zeros(geo.shape))
    return case, geo, p, f0, kappa, target


@pytest.mark.parametrize("grid", GRIDS)
def test_gradient_on_ragged_grids(grid):
    case, geo, p, f0, kappa, target = problem(grid)
    g = gradient(case, kappa, target, 4)
    some = range(0, len(kappa), 3)
    fd = GR.fd_gradient(f0, geo, p, kappa, N_STEPS, target, some, h=1e-5)
    assert np.max(np.abs(fd)) > 0
    assert np.max(np.abs(g[list(some)] - fd)) <= 1e-6 * np.max(np.abs(g))


def test_gradient_with_buffers_beyond_the_pool():
    case, geo, p, f0, kappa, target = problem(GRIDS[3])
    every = (1 << 30) // (9 * 8 * case.mask.size) + 2      # one segment buffer of more than 1 GiB
    assert np.array_equal(gradient(case, kappa, target, N_STEPS), gradient(case, kappa, target, every))


FP32_GRIDS = GRIDS + [   # own nodes of a tile of the FP32 reverse step: 28 x 12
    ((24, 56), (28.0, 12.0), 4.5, (28.0, 20.0), 4.0),   # whole tiles, the body on the corner of four
    ((25, 57), (28.0, 24.0), 4.5, (28.0, 10.0), 6.0),   # one node more each way, the body across the y edge
    ((40, 44), (22.0, 14.0), 7.0, (22.0, 25.0), 8.0),
]


@pytest.mark.parametrize("grid", FP32_GRIDS)
def test_gradient_fp32(grid):
    import torch
    from paper_1908_04443_gb300 import lbmwet as L
    shape, c, R, dc, r = grid
    case = drop_on_cylinder(shape, c, R, dc, r, kappa=0.1)
    geo, _, _ = case.oracle()
    rng = np.random.default_rng(9)
    case.kappa = rng.uniform(0.02, 0.3, len(geo.wall_flat))
    drho = torch.as_tensor(rng.standard_normal(case.mask.size) * (case.mask.reshape(-1) == 0), device="cuda")
    g = {}
    for precision in ("fp64", "fp32"):
        if precision == "fp32":
            case.rho_ref = case.bounds()[0]
        with case.gpu(precision, stream=torch.cuda.current_stream()) as sim:
            L.lbm_record(sim.h, N_STEPS, 4)
            g[precision] = L.lbm_adjoint(sim.h, drho.data_ptr(), len(case.kappa))
            assert sim.check_guards()[0] == 0
    assert np.max(np.abs(g["fp32"] - g["fp64"])) <= 2e-3 * np.max(np.abs(g["fp64"]))
