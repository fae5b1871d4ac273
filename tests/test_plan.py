"""The rules that choose passes of several steps (plan.cuh), compiled for the host.

Tiles: whatever the grid's shape, a launch forms a bounded number of nodes per
multiprocessor and step; a grid of few nodes but many tiles (one node wide, or flat) takes
single steps.

Rows: the parts of a pass cover a plane's rows once, each part (but a plane's only one) keeps
the rows its queues need, and passes are taken only where the nodes formed twice and the
warp slots left idle stay within what they save.
"""

import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SMS = 152

SOURCE = r"""
#include "plan.cuh"
extern "C" int tiles(int dim, int q, int s, int f64, int fixed, int nx, int ny, int nz, int sms, int* out)
{
    const lbms::TileShape t = lbms::tile_shape(dim, q, s, f64 != 0, fixed != 0, nx, ny, nz, sms);
    out[0] = t.x; out[1] = t.y; out[2] = t.z;
    return t.depth;
}
extern "C" void rows(int q, int s, int steps, int nx, int ny, int sms, int* out)
{
    const lbms::RowPlan p = lbms::row_plan(q, s, steps, nx, ny, sms);
    out[0] = p.strips; out[1] = p.segments; out[2] = p.rows;
}
extern "C" int pay(int q, int s, int steps, int nx, int ny, int walls, int sms)
{
    const long long cells = (long long)nx * ny;  // two nodes per thread in single steps (k_step_pair)
    const bool pairs = q <= 7 && s <= 2 && cells >= (1 << 21) && cells % 2 == 0;
    return lbms::rows_pay(q, s, steps, nx, ny, walls != 0, pairs, sms);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC",
                    "-I", os.path.join(ROOT, "paper_1808_06787_gb300", "csrc"), src, "-o", so], check=True)
    return ctypes.CDLL(so)


def tile(lib, dim, q, s, f64, fixed, grid):
    out = (ctypes.c_int * 3)()
    g = tuple(grid) + (1,) * (3 - len(grid))
    return lib.tiles(dim, q, s, f64, fixed, *g, SMS, out), tuple(out)


KINDS = [(1, 3), (2, 4), (2, 5), (2, 9), (3, 6), (3, 7), (3, 15)]


def grids(dim, g):
    shapes = [(1,) * dim, (8192,) + (1,) * (dim - 1), (1,) * (dim - 1) + (8192,), (65536,) + (1,) * (dim - 1)]
    for _ in range(600):
        cells = np.exp(g.uniform(0, np.log(200000)))
        e = g.dirichlet((0.7,) * dim)
        shapes.append(tuple(max(1, int(cells ** v)) for v in e))
    return shapes + [(2 ** 31 - 1,) + (1,) * (dim - 1)]


@pytest.mark.parametrize("f64,fixed", [(0, 0), (1, 1), (1, 0)])
@pytest.mark.parametrize("s", [1, 2, 3, 4, 7])
@pytest.mark.parametrize("dim,q", KINDS)
def test_tiles_form_a_bounded_number_of_nodes(lib, dim, q, s, f64, fixed):
    g = np.random.default_rng([dim, q, s, f64, fixed])
    taken = 0
    for grid in grids(dim, g):
        depth, size = tile(lib, dim, q, s, f64, fixed, grid)
        assert 1 <= depth <= 8
        if depth == 1:
            assert size == (0, 0, 0)
            continue
        taken += 1
        count = np.prod([-(-n // t) for n, t in zip(grid, size)])
        region = np.prod([t + 2 * (depth - 1) for t in size[:dim]])
        assert region <= 512 and all(t == 1 for t in size[dim:])
        # per multiprocessor 1.8 tiles of 400 nodes (FP32) or 1.1 of 308 (FP64); lines 3.4 of 30;
        # or in FP32 planes no more than 7900 units of work a step
        bound = 3.375 * 30 if dim == 1 else (1.1 * 308 if f64 else 1.8 * 400)
        formed = sum(np.prod([t + 2 * m for t in size[:dim]]) for m in range(depth)) / depth
        light = dim == 2 and not f64 and count * formed * (s * q + 4) <= 7900 * SMS
        assert light or count * region <= bound * SMS, (grid, depth, size)
        if s == 3 and q == 9 and size[0] == 16 and size[1] == 16:
            assert light or count <= SMS
        if f64 and not fixed and dim > 1:
            assert depth == 2 and count <= SMS
    assert (taken > 20) == (s <= 3 and not (f64 and s > 2) and (dim < 3 or (q < 15 and s <= 2 and not f64)))


def test_ordinary_grids_keep_their_tiles(lib):
    assert tile(lib, 2, 5, 2, 0, 0, (48, 40)) == (5, (8, 8, 1))
    assert tile(lib, 2, 5, 2, 0, 0, (128, 128)) == (4, (16, 8, 1))
    assert tile(lib, 2, 9, 2, 0, 0, (256, 256)) == (3, (16, 16, 1))
    assert tile(lib, 2, 5, 2, 0, 0, (256, 256)) == (2, (16, 16, 1))
    assert tile(lib, 2, 5, 1, 1, 1, (240, 40)) == (5, (8, 8, 1))
    assert tile(lib, 2, 5, 2, 1, 1, (64, 64)) == (4, (8, 4, 1))
    assert tile(lib, 2, 5, 2, 1, 1, (128, 128))[0] == 1
    assert tile(lib, 3, 7, 2, 0, 0, (24, 16, 12)) == (3, (4, 4, 4))
    for grid in ((65536, 1), (1, 65536), (24576, 1), (2, 32768)):
        assert tile(lib, 2, 5, 2, 0, 0, grid)[0] == 1
    assert tile(lib, 2, 9, 2, 0, 0, (4096, 2))[0] == 1
    for s, q, grid in ((1, 5, (6000, 4)), (1, 5, (5000, 13)), (2, 5, (6000, 4)), (1, 9, (4096, 2)), (2, 9, (20, 1000))):
        assert tile(lib, 2, q, s, 0, 0, grid)[0] > 1
    assert tile(lib, 3, 7, 2, 0, 0, (7168, 1, 1))[0] == 1
    assert tile(lib, 2, 5, 2, 1, 1, (6400, 1))[0] == 1


DEPTH = {1: 3, 2: 3, 3: 2, 4: 2}


def planes(g, count):
    shapes = [(56, 30011), (57, 36792), (64, 32768), (4095, 4097), (2048, 2048), (1 << 20, 24), (24, 1 << 20), (66112, 128)]
    for _ in range(count):
        cells = np.exp(g.uniform(np.log(1 << 18), np.log(1 << 25)))
        a = np.exp(g.uniform(np.log(24), np.log(cells / 24)))
        shapes.append((int(a), int(cells / a)))
    return shapes


@pytest.mark.parametrize("s", [1, 2, 3, 4])
@pytest.mark.parametrize("q", [4, 5, 9])
def test_parts_cover_the_rows_and_pay(lib, q, s):
    g = np.random.default_rng([q, s])
    out = (ctypes.c_int * 3)()
    taken = 0
    for nx, ny in planes(g, 1500):
        for steps in range(2, DEPTH[s] + 1):
            lib.rows(q, s, steps, nx, ny, SMS, out)
            strips, segments, rows = out
            width = 32 - 2 * (steps - 1)
            assert (strips - 1) * width < nx <= strips * width
            assert (segments - 1) * rows < ny <= segments * rows
            assert segments == 1 or rows >= 4 * steps
        if not lib.pay(q, s, DEPTH[s], nx, ny, 0, SMS):
            assert not lib.pay(q, s, DEPTH[s], nx, ny, 1, SMS)
            continue
        taken += 1
        # at most twice the plane's nodes, idle lanes and margins included
        assert strips * 32 * segments * (rows + 2 * (steps - 1)) <= 2.05 * nx * ny
        assert nx >= 56 and ny >= 24
    assert 200 < taken < 1500


def test_narrow_and_flat_planes_take_single_steps(lib):
    """Measured slower in passes than in single steps (1.1 to 1.6 times)."""
    slow = [(4, 2, (64, 32768), 0), (4, 2, (57, 100000), 0), (5, 2, (57, 36792), 0), (5, 2, (64, 32768), 0),
            (5, 2, (20278, 84), 0), (5, 1, (66112, 128), 0), (5, 1, (64, 46048), 1), (5, 3, (64, 15520), 0),
            (9, 4, (73, 42588), 1), (9, 4, (112, 20231), 1), (9, 3, (72, 119535), 1), (9, 2, (37048, 111), 1),
            (4, 4, (64, 8640), 1), (4, 3, (38834, 27), 0)]
    for q, s, (nx, ny), walls in slow:
        assert not lib.pay(q, s, DEPTH[s], nx, ny, walls, SMS), (q, s, nx, ny)
    fast = [(5, 2, (4095, 4097), 1), (9, 4, (2048, 2048), 0), (5, 2, (1448, 1448), 0), (5, 1, (1024, 1024), 0),
            (9, 2, (2048, 2048), 1), (4, 2, (4096, 4096), 0), (5, 4, (2048, 2048), 0)]
    for q, s, (nx, ny), walls in fast:
        assert lib.pay(q, s, DEPTH[s], nx, ny, walls, SMS), (q, s, nx, ny)
