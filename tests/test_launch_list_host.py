"""The work items that a launch of the TMA-staged D3Q19 z-march runs (lbm_d3q19_launch_list, the list lbm_init
builds; host code, no GPU needed), checked against the definitions in the header, restated here with numpy:

* the items of every 32 x 8 column partition the planes [0, nz), each of at least one plane;
* a column cut by the grid's far edge is worked on as a block moved inside the grid that starts on a multiple of
  4 in x and covers all of its own nodes;
* planes within 3 planes (periodic) of one with a solid within 3 nodes (periodic) of that block are on the solid
  path: bounce-back and virtual densities are never skipped;
* a plane on the solid path without need lies in a short run of planes (a cut column's need is taken together
  with its neighbour's, which its block may reach into);
* large grids: cuts at multiples of 32 planes, at most 46 planes a piece, the last layer's bulk pieces in four at
  the end; small ones: near-equal pieces, solid ones first.
"""
import ctypes as C

import numpy as np
import pytest

import workloads as W
from paper_1908_04443_gb300 import lbmwet as L

TX, TY, CH, HALO = 32, 8, 32, 3
SLOTS = 304                     # two CTAs on each of 152 SMs


def _block(bx, by, nx, ny):
    xs, ys = bx * TX, by * TY
    x0 = xs if xs + TX <= nx else (nx - TX + 3) // 4 * 4
    y0 = min(ys, ny - TY)
    assert x0 % 4 == 0 and 0 <= x0 <= xs and x0 + TX >= min(xs + TX, nx) and x0 + TX <= nx + 3
    assert 0 <= y0 <= ys and y0 + TY >= min(ys + TY, ny)
    return x0, y0


def _near(mask, x0, x1, y0, y1):
    """Per plane: within 3 planes of one with a solid within 3 nodes of [x0, x1) x [y0, y1) (periodic)."""
    nz, ny, nx = mask.shape
    xs, ys = np.arange(x0 - HALO, x1 + HALO) % nx, np.arange(y0 - HALO, y1 + HALO) % ny
    near = mask[:, ys][:, :, xs].reshape(nz, -1).any(axis=1)
    return np.array([near[(z + np.arange(-HALO, HALO + 1)) % nz].any() for z in range(nz)])


def _runs(flags):
    out = np.zeros(len(flags), int)
    z0 = 0
    for z in range(1, len(flags) + 1):
        if z == len(flags) or flags[z] != flags[z0]:
            out[z0:z] = z - z0
            z0 = z
    return out


def check(mask, slots):
    nz, ny, nx = mask.shape
    items = L.lbm_d3q19_launch_list(mask, slots)
    gx, gy = -(-nx // TX), -(-ny // TY)
    large = gx * gy * -(-nz // CH) >= 2 * slots
    cols = {}
    for bx, by, z0, z1, s in items.tolist():
        assert 0 <= bx < gx and 0 <= by < gy and 0 <= z0 < z1 <= nz and s in (0, 1)
        cols.setdefault((bx, by), []).append((z0, z1, s))
    assert len(cols) == gx * gy
    for (bx, by), its in cols.items():
        its.sort()
        assert its[0][0] == 0 and its[-1][1] == nz
        assert all(a[1] == b[0] for a, b in zip(its, its[1:])), (bx, by)
        path = np.zeros(nz, bool)
        for z0, z1, s in its:
            path[z0:z1] = s == 1
            assert not large or z1 - z0 <= CH + 2 * 7          # a first and a last piece of up to 7 planes joined
        x0, y0 = _block(bx, by, nx, ny)
        need = _near(mask, x0, x0 + TX, y0, y0 + TY)
        assert not (need & ~path).any(), (bx, by)
        # a cut column together with the neighbour that its block may reach into
        bx0, by0 = bx - (bx * TX + TX > nx and bx > 0), by - (by * TY + TY > ny and by > 0)
        wide = _near(mask, bx0 * TX, bx * TX + TX, by0 * TY, by * TY + TY)
        extra = path & ~wide
        assert not extra.any() or (_runs(wide)[extra] < (8 if large else 4)).all(), (bx, by)
    order = [(z0, by, bx) for bx, by, z0, z1, s in items.tolist()]
    if large:
        zt = (nz - 1) // CH * CH
        n = len(order)
        tail = [k for k in range(n) if items[k, 2] >= zt and not items[k, 4] and items[k, 3] - items[k, 2] < CH]
        m = next((k for k in range(1, n) if order[k] < order[k - 1]), n)   # end of the sorted part
        assert order[:m] == sorted(order[:m])
        assert all(k in tail for k in range(m, n))
        for (bx, by), its in cols.items():
            for (_, z1, s), (_, _, t) in zip(its, its[1:]):
                assert z1 % CH == 0 or s != t or z1 > zt, (bx, by, z1)
    else:
        keys = [(1 - s, z0, by, bx) for bx, by, z0, z1, s in items.tolist()]
        assert keys == sorted(keys)
    return items


SHAPES = [(4, 16, 40), (5, 16, 64), (33, 17, 43), (12, 23, 66), (21, 19, 97), (70, 24, 100), (37, 21, 100), (75, 83, 97),
          (40, 24, 61), (9, 16, 63), (64, 64, 64), (70, 200, 200)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("slots", [1, 8, SLOTS])
@pytest.mark.parametrize("seed", [0, 1])
def test_random_specks(shape, slots, seed):
    rng = np.random.default_rng(seed)
    check((rng.random(shape) < 2e-4).astype(np.uint8), slots)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("slots", [1, SLOTS])
def test_no_solids_no_solid_items(shape, slots):
    assert check(np.zeros(shape, np.uint8), slots)[:, 4].sum() == 0


@pytest.mark.parametrize("where", [(0, 0, 0), (20, 18, 96), (10, 0, 95), (0, 18, 40), (10, 8, 63), (10, 15, 64)])
def test_one_solid_at_an_edge(where):
    """One solid node at the far edges, where the moved blocks and the periodic images meet."""
    mask = np.zeros((21, 19, 97), np.uint8)
    mask[where] = 1
    check(mask, SLOTS)
    check(mask, 1)


def test_spheres():
    check(W.sphere_drop_64().mask(), SLOTS)
    check(W.sphere_fig14(0.2).mask(), SLOTS)
    # as many items as the launch of the 256^3 sphere has CTAs in its profile
    assert len(check(W.c3_sphere_256().mask(), SLOTS)) == 2853


def test_errors():
    mask = np.zeros((40, 16, 64), np.uint8)
    for bad, slots in ((np.zeros((40, 16, 36), np.uint8), 8), (np.zeros((3, 16, 64), np.uint8), 8),
                       (np.zeros((40, 15, 64), np.uint8), 8), (mask, 0), (np.zeros((0, 16, 64), np.uint8), 8)):
        with pytest.raises(L.LbmError):
            L.lbm_d3q19_launch_list(bad, slots)
    lib = L.library()
    n = C.c_int64(-1)
    mp = mask.ctypes.data_as(C.c_void_p)
    assert lib.lbm_d3q19_launch_list(None, 64, 16, 40, 8, None, 0, C.byref(n)) == L.LBM_ERR_ARG
    assert lib.lbm_d3q19_launch_list(mp, 64, 16, 40, 8, None, 0, None) == L.LBM_ERR_ARG
    assert lib.lbm_d3q19_launch_list(mp, 64, 16, 40, 8, None, 0, C.byref(n)) == L.LBM_OK and n.value >= 4
    buf = (C.c_int32 * 5)(*([-7] * 5))
    assert lib.lbm_d3q19_launch_list(mp, 64, 16, 40, 8, buf, 1, C.byref(n)) == L.LBM_ERR_ARG
    assert list(buf) == [-7] * 5
