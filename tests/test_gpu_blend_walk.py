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


def _grads(sc, W, tile):
    r, f, scene, _ = _gpu.run_forward(sc, CAM, tile=tile)
    g = r.run_backward(scene, CAM, f, torch.from_numpy(W.astype(np.float32)).cuda())
    return [t.cpu().numpy().astype(np.float64) for t in g]


@pytest.mark.parametrize("make", [_wide, _spots])
@pytest.mark.parametrize("n", LENGTHS)
def test_backward_walk_lengths(n, make):
    sc = make(n)
    W = np.random.default_rng(3).normal(size=(3, CAM.height, CAM.width)).astype(np.float32)
    ref = oracle.backward(sc, CAM, W.astype(np.float64), mode=1)
    for tile in (8, 16, 32):
        d_ms, d_op, d_col = _grads(sc, W, tile)
        _gpu.grad_close(d_ms[:, :3], ref["d_means"], f"means, tile {tile}")
        _gpu.grad_close(d_ms[:, 3], ref["d_sigma"], f"sigma, tile {tile}")
        _gpu.grad_close(d_op, ref["d_opac"], f"opacity, tile {tile}")
        _gpu.grad_close(d_col, ref["d_color"].reshape(d_col.shape), f"color, tile {tile}")


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_nonfinite_image_gradient_stays_where_it_is_blended(bad):
    # a pixel whose dL/dC is not finite reaches only the Gaussians that it blended:
    # others of the same 8 x 8 block keep the gradients they have without it
    sc = scene_from([[-0.30, 0.0, 0.0], [0.30, 0.0, 0.0], [0.0, 0.3, 0.0]], [0.08] * 3, [0.5] * 3, np.full((3, 3), 0.5))
    cam = scenes.pinhole((0.0, 0.0, -2.0), 16, 16, 16.0)
    W = np.ones((3, 16, 16), np.float32)
    r, f, scene, _ = _gpu.run_forward(sc, cam, tile=16)
    u, v, w2, pmax = f.rec()[:, :4].cpu().numpy().T
    yy, xx = np.mgrid[0:16, 0:16] + 0.5
    inside = w2[:, None, None] * ((xx - u[:, None, None]) ** 2 + (yy - v[:, None, None]) ** 2) <= pmax[:, None, None]
    only0 = inside[0] & ~inside[1] & ~inside[2]
    y, x = np.argwhere(only0)[0]
    base = [t.cpu().numpy() for t in r.run_backward(scene, cam, f, torch.from_numpy(W).cuda())]
    W[:, y, x] = bad
    got = [t.cpu().numpy() for t in r.run_backward(scene, cam, f, torch.from_numpy(W).cuda())]
    assert not np.isfinite(got[2][0]).all()
    for a, b in zip(got, base):
        # two FP32 sums of at most 256 pixels in another association: 256 x 2^-24 of the terms' size
        np.testing.assert_allclose(a[1:], b[1:], rtol=0, atol=2e-5 * np.abs(b).max())
