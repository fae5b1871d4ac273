"""FP64 mole-fraction totals of the integer block sums, and FP64 solves whose nodes leave the
range of the fixed-point collision.

The per-block sums are exact 128-bit integers (units of 2^-118) where every value fits
them, and two-sum pairs otherwise; either way a species' total over the grid must be the
correctly rounded sum of the nodes' mole fractions to within two ulps (the rounding of the
result and of the merged pairs), trace species included.
"""

import math

import numpy as np
import pytest

import synthetic as sy

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1808_06787_gb300 as p

    p.load()


@pytest.mark.parametrize("grid", [(1, 1), (7, 5), (64, 1), (257, 3), (640, 333)])
@pytest.mark.parametrize("kind", ["plain", "trace", "wild"])
def test_totals_are_exact(grid, kind):
    from paper_1808_06787_gb300 import Solver

    s = Solver("D2Q5", sy.random_D(3, seed=1), grid, dtype=torch.float64)
    g = torch.Generator(device="cuda").manual_seed(7)
    f = torch.rand(s.state_shape, dtype=torch.float64, device="cuda", generator=g) * 0.06
    if kind == "trace":
        f[0] *= 10.0 ** (-40.0 * torch.rand(f.shape[2], dtype=torch.float64, device="cuda", generator=g))
    if kind == "wild":
        f[1, 2, ::3] -= 3.0
        f[0, 0, 1::5] += 1e6
    s.set_state_raw(f, 0)
    x = s.moments().double().cpu().numpy().reshape(3, -1)
    for got, row in zip(s.mass(), x):
        want = math.fsum(row)
        assert abs(got - want) <= 2 * np.spacing(abs(want))


@pytest.mark.parametrize("n", [2, 3])
def test_steep_fronts_match_the_oracle(n):
    """Pure gases side by side: the fronts' trace species fall by orders of magnitude from
    node to node, and nodes next to a jump may leave [0, 1] by the scheme's undershoot."""
    import oracle
    from paper_1808_06787_gb300 import Solver

    nx = 48
    x0 = np.zeros((n, 1, 6, nx))
    for s in range(n):
        x0[s, :, :, s * nx // n:(s + 1) * nx // n] = 1.0
    D = sy.random_D(n, seed=9)
    bc = ("noflux", "noflux") + ("periodic",) * 4
    for steps in (1, 40):
        a = Solver("D2Q5", D, (nx, 6), bc=bc, dtype=torch.float64)
        a.set_state(torch.from_numpy(x0).cuda())
        a.step(steps)
        x, J = a.moments(flux=True)
        rx, rJ = oracle.run("D2Q5", D, x0, steps, bc=bc, flux=True)
        assert np.abs(x.cpu().numpy() - rx).max() <= 1e-12
        assert np.abs(J.cpu().numpy() - rJ).max() <= 1e-13
