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


# Ternary D2Q5 nodes that leave the range of the fixed-point collision (populations of two
# species: rest, then opposite pairs)
WILD = {
    "pair below one": [[0.3, 0.99, 0.99, -0.99, -0.99], [0.1, 0.05, 0.05, 0.05, 0.05]],
    "pair above a half": [[0.0, 0.55, 0.02, 0.02, 0.02], [0.1, 0.05, 0.05, 0.05, 0.05]],
    "other species' pair": [[0.1, 0.05, 0.05, 0.05, 0.05], [0.2, -0.97, 0.98, 0.97, -0.96]],
    "mole fraction 1.2": [[0.4, 0.2, 0.2, 0.2, 0.2], [0.0, 0.01, 0.0, 0.01, 0.0]],
    "population above one": [[1.5, -0.2, -0.2, -0.2, -0.2], [0.1, 0.05, 0.05, 0.05, 0.05]],
    "below 2^-900": [[1e-280, 1e-281, 2e-281, 3e-281, 1e-281], [0.1, 0.05, 0.05, 0.05, 0.05]],
    "subnormal species": [[3e-310, 1e-310, 2e-310, 1e-310, 1e-310], [0.1, 0.05, 0.05, 0.05, 0.05]],
    "third species below zero": [[0.25, 0.1, 0.12, 0.1, 0.12], [0.25, 0.12, 0.1, 0.1, 0.1]],
}


def _collide(f, D):
    """The D2Q5 collision with Eq. 3-16's even rates of one ternary node, in FP64."""
    w = np.array([1 / 3] + [1 / 6] * 4)
    x = f.sum(1)
    xi = np.append(x, 1.0 - x.sum())
    B = np.empty((2, 2))
    for i in range(2):
        for j in range(2):
            B[i, j] = (xi[i] * (1 / D[i, 2] - 1 / D[i, j]) if i != j
                       else xi[i] / D[i, 2] + sum(xi[k] / D[i, k] for k in range(3) if k != i))
    odd = np.linalg.solve(B / 2 + 3.0 * np.eye(2), B / 2)
    even = odd.copy()
    for i in range(2):
        even[i, i] = 4 * (odd[i, i] - 1) / (odd[i, i] - 4)
    out = f.copy()
    for a in (1, 3):
        s = even @ (f[:, a] + f[:, a + 1] - 2 * w[a] * x)
        o = odd @ (f[:, a] - f[:, a + 1])
        out[:, a] -= s + o
        out[:, a + 1] -= s - o
    out[:, 0] = x - out[:, 1:].sum(1)
    return out


@pytest.mark.parametrize("grid", [(100, 101), (40, 30), (400, 300)])
@pytest.mark.parametrize("kind", sorted(WILD))
def test_wild_nodes_follow_the_fp64_collision(grid, kind):
    """A uniform periodic field only collides.  Three steps, of two lanes per node, of tiles and
    of one lane per node by the size of the grid, against the collision in numpy; to
    2^-47 of the largest population (a few FP64 roundings of departures up to four), or 64
    subnormal units."""
    from paper_1808_06787_gb300 import Solver

    D = sy.random_D(3, seed=4)
    node = np.array(WILD[kind])
    s = Solver("D2Q5", D, grid, dtype=torch.float64)
    f = torch.from_numpy(node)[:, :, None].expand(s.state_shape).contiguous().cuda()
    s.set_state_raw(f, 0)
    s.step(3)
    want = _collide(_collide(_collide(node, D), D), D)
    got = s.get_state().cpu().numpy()
    for i in range(2):
        scale = max(np.abs(node[i]).max(), np.abs(want[i]).max())
        assert np.abs(got[i] - want[i][:, None]).max() <= max(2.0 ** -47 * scale, 64 * 5e-324)


@pytest.mark.parametrize("faces", ["pp", "ww"])
@pytest.mark.parametrize("grid", [(101, 64), (64, 51)])
def test_isolated_wild_nodes_take_the_same_path_everywhere(grid, faces):
    """Single wild nodes in the warps of an ordinary field, the last one among them: a field
    repeated along a periodic axis until one lane takes a node gives the same populations
    bit for bit as the field alone (two lanes per node, or tiles)."""
    from paper_1808_06787_gb300 import Solver

    nx, ny = grid
    copies = -(-98305 // (nx * ny))
    bc = ("noflux" if faces == "ww" else "periodic",) * 2 + ("periodic",) * 4
    D = sy.random_D(3, seed=4)
    a = Solver("D2Q5", D, (nx, ny), bc=bc, dtype=torch.float64)
    b = Solver("D2Q5", D, (nx, ny * copies), bc=bc, dtype=torch.float64)
    g = np.random.default_rng(8)
    x = g.uniform(0.05, 1.0, (3, nx * ny))
    x /= x.sum(0)
    w = np.array([1 / 3] + [1 / 6] * 4)
    f = w[None, :, None] * x[:2, None, :] * (1 + 0.2 * g.uniform(-1, 1, (2, 5, nx * ny)))
    at = np.concatenate([[0, 15, 16, 17, nx * ny - 1], g.integers(0, nx * ny, 40)])
    for i, c in enumerate(at):
        f[:, :, c] = WILD[sorted(WILD)[i % len(WILD)]]
    f = torch.from_numpy(f).cuda()
    a.set_state_raw(f.contiguous(), 0)
    b.set_state_raw(f.repeat(1, 1, copies).contiguous(), 0)
    for n in (2, 3, 6):
        a.step(n)
        b.step(n)
        want = a.get_state()
        assert torch.isfinite(want).all()
        assert torch.equal(b.get_state(), want.repeat(1, 1, copies))
