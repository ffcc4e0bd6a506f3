"""A pixel that blends one front entry and none of the thousands behind it that its 8 x 8 block
walks: the backward takes its transmittance through all of them (a multiplication by the
approximate reciprocal of 1 each) and must bring it to the front entry unchanged. So the front
entry's gradients equal, bit for bit, those it has alone."""
import numpy as np
import pytest
import torch

from paper_2403_14244_gb300 import scenes

from . import _gpu
from ._tiny import scene_from

pytestmark = pytest.mark.gpu

CAM = scenes.pinhole((0.0, 0.0, -2.0), 8, 8, 8.0)


def _at(u, v, z):
    """World position that projects to pixel position (u, v) at depth z + 2."""
    u, v, z = np.broadcast_arrays(np.asarray(u, float), np.asarray(v, float), np.asarray(z, float))
    return np.stack([(u - 4.0) * (z + 2.0) / 8.0, (v - 4.0) * (z + 2.0) / 8.0, z], -1)


def _front_gradients(n_behind, tile):
    rng = np.random.default_rng(1)
    z = np.sort(rng.uniform(0.0, 0.5, n_behind))
    means = np.concatenate([_at(1.7, 1.4, -0.5)[None], _at(rng.uniform(4.5, 7.5, n_behind), rng.uniform(4.5, 7.5, n_behind), z)])
    sigma = np.concatenate([[0.6 * 1.5 / 8.0], 0.4 * (z + 2.0) / 8.0])         # 0.6 and 0.4 pixels
    opac = np.concatenate([[0.7], rng.uniform(0.0042, 0.005, n_behind)])
    sc = scene_from(means, sigma, opac, np.full((n_behind + 1, 3), 0.5))
    r, f, scene, _ = _gpu.run_forward(sc, CAM, tile=tile, bg=(0.3, 0.2, 0.1))
    contrib = f.n_contrib().cpu().numpy().astype(np.int64)
    G = np.zeros((3, 8, 8), np.float32)
    G[:, 1, 1] = [0.3, -0.7, 1.1]
    grads = r.run_backward(scene, CAM, f, torch.from_numpy(G).cuda())
    return contrib, [g[0].cpu().numpy() for g in grads]


@pytest.mark.parametrize("tile", [8, 16, 32])
def test_transmittance_survives_unblended_entries(tile):
    alone_n, alone = _front_gradients(0, tile)
    n, behind = _front_gradients(4096, tile)
    assert alone_n[1, 1] == n[1, 1] == 1 and n.max() > 4000   # the block's walk is long, the pixel's one entry
    for a, b in zip(behind, alone):
        assert np.abs(b).max() > 0
        np.testing.assert_array_equal(a, b)
