"""The blends' walks at the sizes where batching can go wrong: list lengths around
the staged batch (32), the queue (64) and the segment stride (1024), lists whose
entries mostly miss a block, and blocks cut by the image's edge, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_14244_gb300 import scenes

from . import _gpu
from ._tiny import scene_from

pytestmark = pytest.mark.gpu

LENGTHS = [1, 2, 31, 32, 33, 63, 64, 65, 96, 1023, 1024, 1025, 2100]


def _wide(n, seed=5):
    """n faint Gaussians that cover a 43 x 27 image, so that every pixel walks them all."""
    rng = np.random.default_rng(seed)
    means = rng.uniform(-0.4, 0.4, (n, 3))
    return scene_from(means, rng.uniform(0.2, 0.6, n), rng.uniform(0.02, 0.05, n), rng.uniform(0, 1, (n, 3)))


def _spots(n, seed=6):
    """n small Gaussians: a tile's list mostly misses each of its 8 x 8 blocks."""
    rng = np.random.default_rng(seed)
    means = rng.uniform(-0.7, 0.7, (n, 3))
    return scene_from(means, rng.uniform(0.003, 0.02, n), rng.uniform(0.05, 0.9, n), rng.uniform(0, 1, (n, 3)))


CAM = scenes.pinhole((0.0, 0.0, -2.0), 43, 27, 40.0)


@pytest.mark.parametrize("make", [_wide, _spots])
@pytest.mark.parametrize("n", LENGTHS)
def test_forward_walk_lengths(n, make):
    sc = make(n)
    ref = oracle.render(sc, CAM, mode=1, flag_margin=2e-5)
    images = {}
    for tile in (8, 16, 32):
        images[tile] = _gpu.run_forward(sc, CAM, tile=tile, bg=(0.1, 0.2, 0.3))[3]
        plain = _gpu.run_forward(sc, CAM, tile=tile)[3]
        _gpu.compare_images(plain, ref["img"], ref["flag"], max_flag_frac=0.05)
    # per pixel the walk is the same whatever the binning tile
    np.testing.assert_array_equal(images[8], images[16])
    np.testing.assert_array_equal(images[8], images[32])
