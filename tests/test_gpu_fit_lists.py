"""The 2D experiment's tile lists at their edges, against the oracle: particle counts
around the 2048 that one pass over the particles tests and lists, spread evenly or all
on one tile (lists of several staged batches, the rest of the tiles with empty ones).
Tolerances: a pixel sums at most 4500 FP32 terms of one sign, each within a few 1e-7 of
its value, in index order: 1e-4 of the largest pixel covers the worst sum (4500 x 2^-24
= 2.7e-4 is the bound, its random-walk expectation 4e-6)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_14244_gb300 import igs, scenes
from tests import _gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heap", [False, True])
@pytest.mark.parametrize("k", [255, 257, 2047, 2048, 2049, 4500])
def test_lists_match_oracle(k, heap):
    W, H, D = 70, 50, 9.0
    p = scenes.fit2d_particles(k, 70, 400 + k, sigma=(0.7, 4.0))
    if heap:
        p[:, 0:2] = 16.5 + (p[:, 0:2] - 16.5) * 0.1
    tp = torch.from_numpy(np.ascontiguousarray(p, np.float32)).cuda()
    img = torch.empty((3, H, W), device="cuda")
    igs.fit2d_render(tp, D, img)
    want = oracle.fit2d_render(p, D, W, H)
    np.testing.assert_allclose(img.cpu().numpy(), want, rtol=1e-4, atol=1e-4 * max(1.0, float(np.abs(want).max())))
    G = np.random.default_rng(k).normal(size=(3, H, W)).astype(np.float32)
    grad = torch.full((k, 8), 7.0, device="cuda")
    igs.fit2d_backward(tp, D, torch.from_numpy(G).cuda(), grad)
    got, ref = grad.cpu().numpy(), oracle.fit2d_backward(p, D, G)
    assert np.all(got[:, 6:] == 0)
    for j, name in enumerate(("mu_x", "mu_y", "log_sigma", "A_r", "A_g", "A_b")):
        _gpu.grad_close(got[:, j], ref[:, j], name)
