"""The flag of initial fields whose mole fractions do not sum to one.

LBMS_FLAG_INIT is raised where the FP64 sum of a node's mole fractions is further than
1e-5 from one or not finite.  FP32 fields are tested by an FP32 sum first; the flag must
be that of the FP64 sum on both sides of the bound, for values that cancel, and for
infinities and NaN.
"""

import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NODES = [
    [0.3, 0.3, 0.4], [0.3, 0.3, 0.4 + 4e-6], [0.3, 0.3, 0.4 - 6e-6], [0.3, 0.3, 0.4 + 9.9e-6],
    [0.3, 0.3, 0.4 - 1.02e-5], [0.3, 0.3, 0.4 + 2e-5], [2.0, -1.0, 0.0], [1.9, -1.9, 1.0], [3.0, -2.0, 0.0],
    [1e6, -1e6, 1.0], [16777216.0, -16777216.0, 1.0], [16777216.0, 1.0, -16777216.0], [1e30, -1e30, 1.0],
    [0.0, 0.0, 0.0], [1.0, 0.0, 0.0], [math.nan, 0.5, 0.5], [math.inf, -math.inf, 1.0], [0.5, 0.5, math.nan],
]


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("node", range(len(NODES)))
def test_init_flag_follows_the_fp64_sum(node, batch):
    import paper_1808_06787_gb300 as p
    from paper_1808_06787_gb300.lbms import FLAG_INIT

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    D = np.ones((3, 3)) * 0.1
    x = np.full((3, 1, 5, 7), 1.0 / 3.0, dtype=np.float32)
    x[2] = 1.0 - x[0] - x[1]
    x[:, 0, 2, 3] = np.array(NODES[node], dtype=np.float32)
    v = x[:, 0, 2, 3].astype(np.float64)
    with np.errstate(invalid="ignore"):
        total = (v[0] + v[1]) + v[2]
    bad = not (np.isfinite(v).all() and abs(total - 1.0) <= 1e-5)
    if batch:
        s = p.BatchSolver("D2Q5", [D], [(7, 5)])
        s.set_state([torch.from_numpy(x).cuda()])
    else:
        s = p.Solver("D2Q5", D, (7, 5))
        s.set_state(torch.from_numpy(x).cuda())
    assert bool(s.status() & FLAG_INIT) == bad
