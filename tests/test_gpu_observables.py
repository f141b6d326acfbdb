"""Observables reduction (GPU): the interface-link queue and the several-grid launches against numpy.

The densities alternate at random between the two sides of (rho_l + rho_g) / 2, so that about half of all
links cross it and every warp's queue fills, empties and ends with a remainder.  With no solid and no
step taken the density field is rho0 (to 1e-15) and every count and sum has a direct numpy form.
Tolerances: the mass is a sum of at most 2e5 terms, rounded at 1e-16 each (1e-11 covers any order); the
circle fit solves normal equations of points spread over the whole box, condition below 1e5, from sums
good to 1e-12.
"""
import numpy as np
import pytest

from tests.harness import Case

pytestmark = pytest.mark.gpu


def _case(shape, seed):
    rng = np.random.default_rng(seed)
    d = len(shape)
    probe = Case("D2Q9" if d == 2 else "D3Q19", shape, np.zeros(shape, np.uint8), np.zeros(shape))
    g, l = probe.bounds()
    mid, half = 0.5 * (g + l), 0.5 * (l - g)
    rho = mid + half * rng.uniform(0.2, 0.9, size=shape) * rng.choice([-1.0, 1.0], size=shape)
    hint = tuple(n / 2.0 for n in shape[::-1])
    return Case(probe.lattice, shape, probe.mask, rho, drop_hint=hint), mid


def _reference(case, mid):
    """Mass, extremes, crossing count and the Kasa fit's centre and radius."""
    rho, d = case.rho0, case.rho0.ndim
    n = np.array(rho.shape[::-1], dtype=float)
    idx = np.indices(rho.shape)[::-1].astype(float)
    pts = []
    for ax in range(d):
        rn = np.roll(rho, -1, axis=d - 1 - ax)
        cross = (rho - mid) * (rn - mid) < 0
        p = np.stack([c[cross] for c in idx], axis=1)
        p[:, ax] += ((mid - rho) / (rn - rho))[cross]
        pts.append(p)
    p = np.concatenate(pts) - np.array(case.drop_hint)
    p -= n * np.round(p / n)
    A = np.concatenate([p, np.ones((len(p), 1))], axis=1)
    sol = np.linalg.lstsq(A, -(p ** 2).sum(1), rcond=None)[0]
    c = -0.5 * sol[:d]
    return rho.sum(), rho.max(), rho.min(), len(p), c + np.array(case.drop_hint), np.sqrt(c @ c - sol[d])


def _check(o, ref, d):
    mass, hi, lo, n, c, r = ref
    assert o.n_interface == n
    assert abs(o.mass - mass) < 1e-11 * mass
    assert abs(o.rho_max - hi) < 1e-14 and abs(o.rho_min - lo) < 1e-14
    assert np.max(np.abs(np.array(o.drop_center[:d]) - c)) < 1e-7 * r
    assert abs(o.drop_radius - r) < 1e-7 * r


@pytest.mark.parametrize("shape", [(5, 7), (8, 32), (33, 31), (300, 257), (4, 5, 6), (20, 19, 67)])
def test_observables_of_random_crossings(shape):
    case, mid = _case(shape, 11)
    with case.gpu("fp64") as sim:
        o, rho, _ = sim.observables(fields=True)
    assert np.max(np.abs(rho - case.rho0)) < 1e-15 * 4
    _check(o, _reference(case, mid), len(shape))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_batch_observables_equal_single_grids(precision):
    """40 grids (more than one load of the grid table per warp) of 1 to 100 tiles."""
    from paper_1908_04443_gb300 import lbmwet as L
    rng = np.random.default_rng(3)
    cases = [_case(tuple(int(v) for v in rng.integers(4, 120, size=2)), i)[0] for i in range(40)]
    cfgs, single = [], []
    for cs in cases:
        cs.rho_ref = cs.bounds()[0] if precision == "fp32" else 0.0
        with cs.gpu(precision) as sim:
            cfgs.append(sim.cfg)
            single.append(sim.observables(fields=True))
    b = L.lbm_batch_init(cfgs, [cs.mask for cs in cases], [cs.rho0 for cs in cases])
    try:
        rhos = [np.zeros(cs.mask.size) for cs in cases]
        us = [np.zeros(2 * cs.mask.size) for cs in cases]
        got = L.lbm_batch_observables_fields(b, rhos, us)
    finally:
        L.lbm_batch_destroy(b)
    for o, r, u, (so, sr, su) in zip(got, rhos, us, single):
        assert np.array_equal(r, sr.reshape(-1)) and np.array_equal(u, su.reshape(-1))
        assert (o.mass, o.rho_max, o.rho_min, o.u_max, o.n_interface) == \
            (so.mass, so.rho_max, so.rho_min, so.u_max, so.n_interface)
        assert tuple(o.drop_center[:2]) == tuple(so.drop_center[:2]) and o.drop_radius == so.drop_radius
