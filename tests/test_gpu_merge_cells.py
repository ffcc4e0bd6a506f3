"""Merged cells at the edges of the two lists (at most eight members, four cells to a
warp; more, a warp each, in runs of 32) and of the sorted items (the last cell ends at
the end of the array), every colour row length, bounds as for any merge. Then
keys that three of the sort's digits hold, and the first that need the fourth."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_merge3d import LO, _compare, _run, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sh", [-1, 0, 1, 2, 3])
@pytest.mark.parametrize("sizes", [[2], [8], [9], [1, 2, 7, 8, 9, 31, 32, 33, 64, 65], [2] * 129 + [8] * 3 + [40],
                                   [3, 1, 1, 5] * 100])
def test_cell_sizes(sizes, sh):
    C = 3 if sh < 0 else 3 * (sh + 1) ** 2
    h, n = 0.05, sum(sizes)
    rng = np.random.default_rng(n + C)
    p, m, v = _state(n, C, 3000 + n, 1)
    cell = np.repeat(rng.permutation(30 ** 3)[: len(sizes)], sizes)
    xyz = np.stack([cell % 30, cell // 30 % 30, cell // 900], 1)
    p[0][:, :3] = -1.0 + h * (xyz + rng.uniform(0.1, 0.9, (n, 3)))
    p[1][:] = rng.normal(0, 1.5, n)
    order = rng.permutation(n)
    p, m, v = ([a[order] for a in g] for g in (p, m, v))
    want = oracle.merge3d(p, m, v, 1, LO, h, 1e9)
    k, got = _run(p, m, v, sh, 1, h, 1e9)
    assert k == want[0][0].shape[0] == len(sizes)
    assert _compare(got, want, 1, h, p) == sum(s > 1 for s in sizes)


@pytest.mark.parametrize("top", [254, 255, 256, 1023])
def test_cell_keys_at_the_third_digit(top):
    """Pairs in the cells (0, 0, 0), (top, top, top) and along each axis at `top`, among Gaussians that
    are not eligible (whose key shares its low digits with cell (255, 255, 255))."""
    n, C, h = 400, 12, 2.0 ** -9
    rng = np.random.default_rng(top)
    p, m, v = _state(n, C, 4000 + top, 1)
    cells = np.array([[0, 0, 0], [top, top, top], [top, 0, 0], [0, top, 0], [0, 0, top], [top, top, 0]])
    xyz = cells[rng.integers(0, len(cells), n)]
    p[0][:, :3] = -1.0 + h * (xyz + rng.uniform(0.2, 0.8, (n, 3)))
    p[1][:] = rng.normal(0, 1.5, n)
    p[1][rng.random(n) < 0.5] = -60.0              # below the floor: kept
    want = oracle.merge3d(p, m, v, 1, LO, h, 1e9)
    k, got = _run(p, m, v, 1, 1, h, 1e9)
    assert k == want[0][0].shape[0]
    assert _compare(got, want, 1, h, p) == len(cells)
