"""Row pitches of the distribution buffers (csrc/layout.h): the kernels other than the TMA-staged z-march form
direction * stride + node in 32 bits, so the pitch must keep that in range on every grid that lbm_init accepts
(up to 2^31 / 19 nodes).  Host arithmetic only: no such grid is allocated or stepped.
"""
import ctypes as C
import os
import random
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
LIMIT = 2 ** 31 // 19          # nodes that lbm_init accepts
INT_MAX = 2 ** 31 - 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    out = str(tmp_path_factory.mktemp("layout") / "liblayout_test.so")
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-o", out,
                        os.path.join(HERE, "native", "layout_shim.cpp")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(out)


def grids_3d():
    """(nx, ny, nz) next to the limit: thin, narrow, shallow, cubic, and random ones."""
    out = [(1, 5400, 5400), (37, 1700, 1700), (37, 1200, 2500), (5, 4000, 4000), (481, 485, 483), (481, 481, 481),
           (39, 1000, 2898), (2000, 15, 3767), (6001, 6001, 3), (41, 16, 172294), (113025455, 1, 1)]
    rng = random.Random(7)
    for _ in range(2000):
        nx = int(2 ** rng.uniform(0, 11))
        ny = int(2 ** rng.uniform(0, 13))
        out.append((nx, ny, max(1, LIMIT // (nx * ny))))
    return [g for g in out if g[0] * g[1] * g[2] <= LIMIT]


@pytest.mark.parametrize("fp32", [True, False])
@pytest.mark.parametrize("kernel", ["auto", "pair", "tile"])
def test_3d_offsets_fit_their_type(lib, fp32, kernel):
    for nx, ny, nz in grids_3d():
        march = fp32 and kernel == "auto" and bool(lib.layout_marches(nx, ny, nz))
        fp = lib.layout_pitch(3, int(march), nx, ny)
        assert nx <= fp < nx + 4
        if march:
            assert fp % 4 == 0                                   # 64-bit direction offsets; rows TMA can address
            assert fp * ny * nz <= INT_MAX                       # 32-bit within one direction
        else:
            assert 19 * fp * ny * nz <= INT_MAX, (nx, ny, nz)


def test_2d_offsets_fit(lib):
    """Narrow, tall grids (batches, the y-march and the set-up take them) as well as ordinary ones, whose rows
    stay padded to 32 nodes."""
    rng = random.Random(8)
    grids = [(1, LIMIT), (7, LIMIT // 7), (15, LIMIT // 15), (16, LIMIT // 16), (31, LIMIT // 31), (33, LIMIT // 33),
             (7, 7456540), (7, 7456541), (600, 400), (10630, 10630)]
    for _ in range(2000):
        nx = int(2 ** rng.uniform(0, 14))
        grids.append((nx, max(1, int(LIMIT / nx * rng.choice([1.0, 1.0, rng.random()])))))
    for nx, ny in grids:
        assert nx * ny <= LIMIT
        fp = lib.layout_pitch(2, 0, nx, ny)
        padded = (nx + 31) // 32 * 32
        assert 9 * fp * ny <= INT_MAX, (nx, ny)
        assert fp == (padded if 9 * padded * ny <= INT_MAX else nx)
