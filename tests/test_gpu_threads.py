"""Solvers of one kernel with tiles of different sizes, stepped by threads at the same time.

Each pass over tiles takes its own amount of shared memory.  Calls of ever new lengths are
launched from several threads, each with its own solver and stream; every call has to
succeed, and the states have to be those of single steps, bit for bit.
"""

import threading

import pytest

import synthetic as sy

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_tiles_of_different_sizes_from_several_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_06787_gb300 import Solver

    grids = [(90, 90), (150, 140), (180, 190), (60, 130)]  # 5, 4, 3 and 5 steps a pass
    solvers, twins, streams = [], [], []
    for i, grid in enumerate(grids):
        streams.append(torch.cuda.Stream())
        pair = [Solver("D2Q9", sy.random_D(4, seed=i), grid, stream=st) for st in (streams[-1], None)]
        x = torch.rand(pair[0].field_shape, device="cuda", dtype=torch.float64) + 0.05
        x = (x / x.sum(0, keepdim=True)).float()
        torch.cuda.synchronize()
        for s in pair:
            s.set_state(x)
        solvers.append(pair[0])
        twins.append(pair[1])
    torch.cuda.synchronize()
    lengths = [n for _ in range(6) for n in range(4, 40)]
    errors = []

    def work(s):
        try:
            for n in lengths:
                s.step(n)
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in solvers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]
    for s, b in zip(solvers, twins):
        out = torch.empty((64,) + tuple(b.state_shape), device="cuda")
        f, left, done = b.get_state(), sum(lengths), 0
        while left:
            m = min(left, 64)
            b.recompute(f, done, m, out)
            f, left, done = out[m - 1].clone(), left - m, done + m
        torch.cuda.synchronize()
        assert torch.equal(s.populations(), f)
