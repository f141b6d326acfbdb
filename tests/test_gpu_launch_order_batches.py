"""The launch order of batches and of the adjoint: as in test_gpu_launch_order, calls issued without a pause give,
bit for bit, what they give with a device synchronisation after every call.  Batches of the FP32 pair kernel (tile
claims counted on the device and reset by the launch before), the FP32 and FP64 tile kernels, the y-march, and groups
of different kernels on branches; the adjoint with its recomputation on a second stream, for checkpoint distances
that divide the steps and that do not, one segment and several, repeated.
"""
import numpy as np
import pytest

from tests.harness import drop_on_cylinder

pytestmark = pytest.mark.gpu

GRIDS = [((40, 48), (24.0, 14.0), 6.0, (24.0, 28.0), 7.0), ((150, 131), (65.0, 50.0), 20.0, (65.0, 95.0), 24.0),
         ((64, 97), (48.0, 20.0), 8.0, (48.0, 38.0), 9.0)]


def _sequence(precision, kinds, sync):
    import torch
    from paper_1908_04443_gb300 import lbmwet as L
    cases = [drop_on_cylinder(*g, kappa=0.08 + 0.02 * i) for i, g in enumerate(GRIDS)]
    cfgs = []
    for cs in cases:
        if precision == "fp32":
            cs.rho_ref = cs.bounds()[0]
        with cs.gpu(precision) as sim:
            cfgs.append(sim.cfg)
    b = L.lbm_batch_init(cfgs, [cs.mask for cs in cases], [cs.rho0 for cs in cases], None)
    out = []
    try:
        L.lbm_batch_set_kernels(b, kinds)
        hs = [L.lbm_batch_handle(b, i) for i in range(len(cases))]
        rho = [torch.zeros(cs.mask.size, dtype=torch.float64, device="cuda") for cs in cases]
        u = [torch.zeros(2 * cs.mask.size, dtype=torch.float64, device="cuda") for cs in cases]
        torch.cuda.synchronize()

        def call(f, *a):
            r = f(*a)
            if sync:
                torch.cuda.synchronize()
            return r

        for k, n in enumerate((1, 1, 1, 16, 2, 33, 1)):
            call(L.lbm_batch_enqueue_steps, b, n)
            for h, r, v in zip(hs, rho, u):
                call(L.lbm_fields_device, h, r.data_ptr(), v.data_ptr())
            if k in (2, 5):
                out += [np.array([(o.mass, o.rho_max, o.rho_min, o.u_max, o.theta_deg, o.n_interface)
                                  for o in call(L.lbm_batch_observables, b)])]
        L.lbm_batch_step(b, 1)
        torch.cuda.synchronize()
        for h, r, v, cs in zip(hs, rho, u, cases):
            out += [r.cpu().numpy(), v.cpu().numpy(), L.lbm_get_state(h, 9, cs.mask.size)]
    finally:
        L.lbm_batch_destroy(b)
    return out


@pytest.mark.parametrize("precision,kinds", [("fp32", ["pair"] * 3), ("fp32", ["tile"] * 3), ("fp64", ["tile"] * 3),
                                             ("fp64", ["ymarch"] * 3), ("fp32", ["pair", "ymarch", "tile"]),
                                             ("fp64", ["tile", "ymarch", "tile"])])
def test_batch_calls_in_a_row_as_one_by_one(precision, kinds):
    for a, b in zip(_sequence(precision, kinds, False), _sequence(precision, kinds, True)):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("grid", GRIDS[:2])
def test_adjoint_for_every_checkpoint_distance(precision, grid):
    """The gradient does not depend on where the trajectory is recomputed from, nor on what ran before."""
    import torch
    from paper_1908_04443_gb300 import lbmwet as L
    case = drop_on_cylinder(*grid, kappa=0.1)
    if precision == "fp32":
        case.rho_ref = case.bounds()[0]
    geo, _, _ = case.oracle()
    rng = np.random.default_rng(3)
    case.kappa = rng.uniform(0.02, 0.3, len(geo.wall_flat))
    drho = torch.as_tensor(rng.standard_normal(case.mask.size), device="cuda")
    out = []
    for every in (23, 4, 1, 11, 22, 23):
        with case.gpu(precision, stream=torch.cuda.current_stream()) as sim:
            L.lbm_record(sim.h, 23, every)
            out.append(L.lbm_adjoint(sim.h, drho.data_ptr(), len(case.kappa)))
            out.append(L.lbm_adjoint(sim.h, drho.data_ptr(), len(case.kappa)))
    assert np.max(np.abs(out[0])) > 0
    for g in out[1:]:
        assert np.array_equal(out[0], g)
