"""Calls captured into a caller's CUDA graph.

A graph of step(n) with n even ends in the buffer and the step counter it began with, so
that every launch of it advances n steps, also where a launch of a kernel takes several
steps.  The state after some launches is compared bit for bit with one that took the steps
one call at a time.  Calls of even lengths in rotation outside capture are compared too:
they replay graphs kept by length and buffer.
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


CASES = [  # lattice, species, grid, dtype, steps: tiles, rows, lines, single steps
    ("D2Q5", 3, (48, 40), torch.float32, (8, 20, 70)), ("D2Q5", 2, (100, 40), torch.float64, (10, 18)),
    ("D2Q5", 3, (60, 50), torch.float64, (10, 12)), ("D3Q7", 3, (18, 17, 16), torch.float32, (4, 6)),
    ("D2Q5", 3, (1500, 1400), torch.float32, (6, 12)), ("D2Q5", 5, (1100, 1200), torch.float32, (4, 8)),
    ("D1Q3", 3, (20000,), torch.float32, (10, 70)), ("D2Q5", 3, (120, 110), torch.float64, (4,)),
]


def _pair(lattice, n, grid, dtype, stream):
    from paper_1808_06787_gb300 import Solver

    g = torch.Generator(device="cuda").manual_seed(2)
    a, b = (Solver(lattice, sy.random_D(n, seed=6), grid, dtype=dtype, stream=st) for st in (stream, None))
    x = torch.rand(a.field_shape, device="cuda", dtype=torch.float64, generator=g) + 0.05
    x = (x / x.sum(0, keepdim=True)).to(dtype)
    torch.cuda.synchronize()
    a.set_state(x)
    b.set_state(x)
    return a, b


@pytest.mark.parametrize("first", [0, 1, 2])
@pytest.mark.parametrize("lattice,n,grid,dtype,lengths", CASES)
def test_replays_of_a_captured_call_advance(lattice, n, grid, dtype, lengths, first):
    for steps in lengths:
        stream = torch.cuda.Stream()
        a, b = _pair(lattice, n, grid, dtype, stream)
        a.step(first)
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            a.step(steps)
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        for _ in range(first + 3 * steps):
            b.step(1)
        torch.cuda.synchronize()
        assert torch.equal(a.populations(), b.populations()), steps
        xa, Ja = a.moments(flux=True)
        torch.cuda.synchronize()
        xb, Jb = b.moments(flux=True)
        torch.cuda.synchronize()
        assert torch.equal(xa, xb) and torch.equal(Ja, Jb)


def test_replays_of_a_captured_batch_call_advance():
    from paper_1808_06787_gb300 import BatchSolver

    grids = [(251 - i, 240 + i) for i in range(74)]
    Ds = [sy.random_D(3, seed=i) for i in range(len(grids))]
    g = torch.Generator(device="cuda").manual_seed(3)
    fields = []
    for nx, ny in grids:
        x = torch.rand((3, 1, ny, nx), device="cuda", dtype=torch.float64, generator=g) + 0.05
        fields.append((x / x.sum(0, keepdim=True)).float())
    for steps in (6, 12, 40):
        stream = torch.cuda.Stream()
        a, b = BatchSolver("D2Q5", Ds, grids, stream=stream), BatchSolver("D2Q5", Ds, grids)
        assert a.step_launches(steps) < steps, "not in passes of several steps"
        torch.cuda.synchronize()
        a.set_state(a.pack(fields))
        b.set_state(b.pack(fields))
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            a.step(steps)
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        for _ in range(3 * steps):
            b.step(1)
        torch.cuda.synchronize()
        xa, Ja = a.moments(flux=True)
        torch.cuda.synchronize()
        xb, Jb = b.moments(flux=True)
        torch.cuda.synchronize()
        assert torch.equal(xa, xb) and torch.equal(Ja, Jb)


def test_lengths_in_rotation():
    """Four lengths of an odd number of launches each, from both buffers in turn."""
    a, b = _pair("D2Q5", 3, (48, 40), torch.float32, None)
    total = 0
    for _ in range(3):
        for steps in (8, 10, 18, 20):
            assert a.step_launches(steps) % 2 == 1
            a.step(steps)
            total += steps
    for _ in range(total):
        b.step(1)
    assert torch.equal(a.populations(), b.populations())
