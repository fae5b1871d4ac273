"""Passes of several steps (fused.cuh, tile.cuh) against the single steps.

lbms_step takes large planes, lines and small grids several steps at a time; lbms_recompute always
launches single steps.  Both use the same node functions and rounding keys, so the
populations must be equal bit for bit, at every edge: strips that end inside the grid, a
last part with fewer rows, walls and wraps on every face, step counts that leave
remainders, and rows of odd length.
"""

import numpy as np
import pytest

import synthetic as sy

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1808_06787_gb300 as p

    p.load()


def _solver(lattice, n, grid, faces, relax, seed=5, dtype=torch.float32):
    from paper_1808_06787_gb300 import Solver

    kind = {"p": "periodic", "w": "noflux", "d": "dirichlet"}
    held = {f: np.full(n, 1.0 / n) + np.linspace(-0.1, 0.1, n) * (1 - 2 * (f % 2)) for f in range(6) if faces[f] == "d"}
    s = Solver(lattice, sy.random_D(n, seed=seed), grid, bc=[kind[c] for c in faces], relax=relax, dtype=dtype,
               boundary=held, reference=np.full(n, 1.0 / n) if relax == "frozen" else None)
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand(s.field_shape, device="cuda", dtype=torch.float64, generator=g) + 0.05
    s.set_state((x / x.sum(0, keepdim=True)).to(dtype))
    return s


CASES = [  # lattice, species, grid, faces
    ("D2Q5", 3, (4099, 401), "wwpppp"), ("D2Q5", 3, (56, 30011), "pppppp"), ("D2Q5", 3, (1251, 1258), "wwwwpp"),
    ("D2Q5", 3, (65537, 24), "ppwwpp"), ("D2Q5", 2, (1025, 1027), "wwwwpp"), ("D2Q4", 3, (1280, 1236), "pppppp"),
    ("D2Q4", 2, (57, 18403), "wwwwpp"), ("D2Q9", 2, (1024, 1024), "wwwwpp"), ("D2Q9", 3, (1053, 1000), "wwwwpp"),
    ("D2Q9", 3, (1000, 1053), "ppwwpp"), ("D2Q9", 4, (701, 751), "wwpppp"), ("D2Q9", 5, (729, 720), "wwwwpp"),
    ("D2Q5", 5, (1111, 480), "ppwwpp"), ("D2Q5", 4, (56, 9400), "wwpppp"),
    ("D1Q3", 3, (1,), "pppppp"), ("D1Q3", 2, (7,), "wwpppp"), ("D1Q3", 3, (112,), "wwpppp"),
    ("D1Q3", 3, (113,), "pppppp"), ("D1Q3", 2, (127,), "pppppp"), ("D1Q3", 3, (100003,), "wwpppp"),
    ("D1Q3", 3, (8193,), "pppppp"), ("D1Q3", 2, (8300,), "wwpppp"),
]
TILED = [  # small grids: tiles, margins that wrap around, walls, Dirichlet faces, both dtypes
    ("D1Q3", 4, (8192,), "wwpppp", "f32"), ("D1Q3", 3, (5,), "pppppp", "f64"), ("D1Q3", 2, (333,), "ddpppp", "f64"),
    ("D2Q5", 3, (1, 1), "pppppp", "f32"), ("D2Q5", 3, (3, 2), "wwpppp", "f32"), ("D2Q5", 3, (48, 40), "wwwwpp", "f32"),
    ("D2Q5", 2, (65, 63), "ddwwpp", "f32"), ("D2Q5", 4, (129, 127), "ppddpp", "f32"), ("D2Q9", 3, (7, 100), "wwwwpp", "f32"),
    ("D2Q9", 2, (256, 255), "pppppp", "f32"), ("D2Q9", 4, (200, 150), "wwddpp", "f32"), ("D2Q4", 3, (250, 260), "wwpppp", "f32"),
    ("D2Q5", 3, (255, 257), "ppwwpp", "f32"), ("D2Q5", 2, (240, 40), "ddpppp", "f64"), ("D2Q5", 2, (141, 143), "wwwwpp", "f64"),
    ("D2Q5", 3, (64, 64), "ddddpp", "f64"), ("D2Q9", 3, (79, 81), "wwwwpp", "f64"), ("D2Q4", 3, (13, 9), "pppppp", "f64"),
    ("D3Q7", 3, (18, 17, 16), "wwwwww", "f32"), ("D3Q6", 2, (5, 3, 2), "pppppp", "f32"), ("D3Q7", 2, (25, 22, 21), "ddwwpp", "f32"),
]


@pytest.mark.parametrize("relax", ["magic", "srt", "frozen"])
@pytest.mark.parametrize("lattice,n,grid,faces,dtype", TILED)
def test_tiled_passes_equal_single_steps(lattice, n, grid, faces, dtype, relax):
    """Grids that leave most of the chip idle take tiles with margins, several steps a pass."""
    _compare(lattice, n, grid, faces, relax, {"f32": torch.float32, "f64": torch.float64}[dtype])


@pytest.mark.parametrize("relax", ["magic", "srt"])
@pytest.mark.parametrize("lattice,n,grid,faces", CASES)
def test_fused_passes_equal_single_steps(lattice, n, grid, faces, relax):
    _compare(lattice, n, grid, faces, relax, torch.float32)


def _compare(lattice, n, grid, faces, relax, dtype):
    a = _solver(lattice, n, grid, faces, relax, dtype=dtype)
    for steps in (2, 3, 4, 9, 20):
        assert a.step_launches(steps) < steps or steps == 2, "not fused"
        f0, t0 = a.get_state(), a.steps_done
        out = torch.empty((steps,) + a.state_shape, device="cuda", dtype=dtype)
        a.recompute(f0, t0, steps, out)
        a.step(steps)
        assert torch.equal(a.get_state(), out[-1]), steps
        if steps == 9:  # the fluxes need the state one step back
            J = a.moments(flux=True)[1]
            b = _solver(lattice, n, grid, faces, relax, dtype=dtype)
            b.set_state_raw(out[-2].contiguous(), t0 + steps - 1)
            b.step(1)
            assert torch.equal(b.moments(flux=True)[1], J)
    # a long call goes through the captured pieces of 32 .. 2 steps
    f0, t0 = a.get_state(), a.steps_done
    a.step(71)
    out = torch.empty((71,) + a.state_shape, device="cuda", dtype=dtype) if np.prod(a.state_shape) < 1 << 22 else None
    if out is not None:
        a.recompute(f0, t0, 71, out)
        assert torch.equal(a.get_state(), out[-1])
    assert a.steps_done == t0 + 71


def test_launch_counts():
    a = _solver("D2Q5", 3, (512, 512), "pppppp", "magic")  # a plane of middle size takes single steps
    assert [a.step_launches(n) for n in (0, 1, 2, 20, 71)] == [0, 1, 2, 20, 71]
    b = _solver("D1Q3", 3, (50000,), "pppppp", "magic")  # eight at a time, the last by itself
    assert [b.step_launches(n) for n in (1, 2, 9, 10, 20)] == [1, 2, 2, 3, 4]
    assert b.step_launches(71) == 1 + 2 * 4 + 1 + 1


@pytest.mark.parametrize("lattice,n", [("D2Q5", 3), ("D2Q5", 2), ("D2Q4", 3)])
@pytest.mark.parametrize("relax", ["magic", "srt"])
def test_fused_batches_equal_single_steps(lattice, n, relax):
    """A batch large enough for passes of several steps, with instances of every awkward
    shape in it, under the streamed candidate (passes) and the one-node candidate (single
    steps), over runs that leave remainders: fields, fluxes and masses are equal bit for bit."""
    from paper_1808_06787_gb300 import BatchSolver

    grids = [(1, 1), (2, 1), (1, 2), (33, 17), (50, 3), (5, 91), (28, 96), (29, 97), (56, 193), (257, 3)]
    grids += [(251 - i, 240 + i) for i in range(72)]
    assert sum(a * b for a, b in grids) >= 1 << 22
    kinds = [("periodic",) * 6, ("noflux", "noflux") + ("periodic",) * 4, ("periodic",) * 2 + ("noflux",) * 2 + ("periodic",) * 2,
             ("noflux",) * 4 + ("periodic",) * 2]
    bcs = [kinds[i % 4] for i in range(len(grids))]
    Ds = [sy.random_D(n, seed=100 + i) for i in range(len(grids))]
    b = BatchSolver(lattice, Ds, grids, bcs=bcs, relax=relax)
    g = torch.Generator(device="cuda").manual_seed(3)
    fields = []
    for nx, ny in grids:
        x = torch.rand((n, 1, ny, nx), device="cuda", dtype=torch.float64, generator=g) + 0.05
        fields.append((x / x.sum(0, keepdim=True)).float())
    got = {}
    for candidate in (7, 0):
        b.set_schedule(candidate)
        b.set_state(b.pack(fields))
        for steps in (1, 2, 3, 20, 40):
            launches = b.step_launches(steps)
            assert launches == steps if candidate == 0 or steps < 3 else launches < steps
            b.step(steps)
        x, J = b.moments(flux=True)
        got[candidate] = (x, J, b.mass(), b.steps_done)
    assert torch.equal(got[7][0], got[0][0]) and torch.equal(got[7][1], got[0][1])
    assert np.array_equal(got[7][2], got[0][2]) and got[7][3] == got[0][3] == 66
