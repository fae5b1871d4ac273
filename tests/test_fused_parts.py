"""Host replay of the parts of the passes of several steps (fused.cuh).

A plane is cut into strips of 32 - 2 (K - 1) columns and parts of rows; a line into
runs of 128 - 2 K nodes.  The rules are replayed here: every node is stored by exactly
one part, and every part but the last keeps at least the rows its queues need.
"""

import numpy as np
import pytest


def cut(n, wave, pair, good, least):
    waves = min(int((n // good) / wave), 4)
    if waves < 2:
        waves = 2 if n // pair >= 2.0 * wave else 1
    s = max(min(int(waves * wave), n // least), 1)
    rows = -(-n // s)
    return -(-n // rows), rows


@pytest.mark.parametrize("steps", [2, 3])
@pytest.mark.parametrize("blocks", [2, 3, 4, 5])
@pytest.mark.parametrize("pair,good", [(16, 48), (32, 48), (80, 80)])
def test_planes_are_covered_once(steps, blocks, pair, good):
    W, H = 32 - 2 * (steps - 1), steps - 1
    g = np.random.default_rng(steps * 10 + blocks)
    shapes = [(56, 24), (56, 1 << 20), (1 << 20, 24), (4095, 4097), (8192, 8192), (28, 2000)]
    shapes += [tuple(int(v) for v in np.exp(g.uniform(np.log(24), np.log(40000), 2))) for _ in range(200)]
    for nx, ny in shapes:
        strips = -(-nx // W)
        segments, rows = cut(ny, 152 * blocks * 4 / strips, pair, good, 4 * steps)
        cols = np.zeros(nx, dtype=int)
        for t in {0, 1, strips // 2, strips - 2, strips - 1} if strips > 6 else range(strips):
            X = t * W - H + np.arange(32)
            mine = X[(np.arange(32) >= H) & (np.arange(32) < 32 - H) & (X < nx)]
            assert mine.size and mine.min() >= 0
            np.add.at(cols, mine, 1)
        assert cols.max() == 1 and (strips > 6 or cols.min() == 1)
        y0 = np.arange(segments) * rows
        y1 = np.minimum(y0 + rows, ny)
        assert y0[-1] < ny and (y1 > y0).all() and (y1 - y0).sum() == ny
        assert segments == 1 or rows >= 4 * steps or rows * segments >= ny


@pytest.mark.parametrize("depth", range(2, 9))
@pytest.mark.parametrize("nx", [1, 7, 31, 111, 112, 113, 128, 5000, 100003])
def test_lines_are_covered_once(depth, nx):
    W = 128 - 2 * depth
    hits = np.zeros(nx, dtype=int)
    for part in range(-(-nx // W)):
        first = part * W
        X = first - depth + np.arange(128)
        np.add.at(hits, X[(X >= first) & (X < min(first + W, nx))], 1)
    assert (hits == 1).all()
