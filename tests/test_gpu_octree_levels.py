"""The Octree initialisation at the seams of its parts, bit for bit against the oracle:
few levels (all sums in the one CTA of the top levels, some there, some above), shares
of the selection's CTAs that are empty or partly filled, budgets inside the first and
the last digits, and leaves of 4095, 4096 and 4097 points, around which the mean colour
goes from FP32 to FP64 steps."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_14244_gb300 import igs

pytestmark = pytest.mark.gpu

LO = (-1.0, -1.0, -1.0)


def _same(p, c, L, k_max, sh, mode):
    want = oracle.octree_init(p, c, LO, 2.0, L, k_max, opacity=0.4, sh_degree=sh, param_mode=mode)
    got = igs.octree_init(torch.from_numpy(p).cuda(), torch.from_numpy(c).cuda(), LO, 2.0, L, k_max, opacity=0.4,
                          sh_degree=sh, param_mode=mode)
    assert got[0].shape[0] == want[0].shape[0]
    for g, w in zip(got, want):
        np.testing.assert_array_equal(g.cpu().numpy(), w)


@pytest.mark.parametrize("L", [1, 2, 3, 4, 6])
@pytest.mark.parametrize("k_max", [2, 9, 333, 3999])
def test_levels(L, k_max):
    rng = np.random.default_rng(10 * L + k_max)
    p = (rng.normal(0, 0.3, (4000, 3))).astype(np.float32)
    c = rng.uniform(-0.1, 1.1, (4000, 3)).astype(np.float32)
    _same(p, c, L, k_max, -1 if k_max % 2 else 1, L % 2)


@pytest.mark.parametrize("sh", [-1, 0])
@pytest.mark.parametrize("n", [4095, 4096, 4097, 9001])
def test_points_of_a_leaf(n, sh):
    rng = np.random.default_rng(n)
    p = rng.uniform(-1, 0, (n + 3, 3)).astype(np.float32)
    p[n:] += 1.0                                    # three points in the opposite octant
    c = rng.uniform(0, 1, (n + 3, 3)).astype(np.float32)
    c[: n // 3] = 0.0
    _same(p, c, 1, 2, sh, 0)                        # one split: the octants are leaves
