"""Where the forward blend cuts a block's walk for the backward: list lengths around the stride of
frames of few blocks (256), lists of more than 64 segments of it and of more than the room for short
segments, blocks whose first blends lie far down the list, and both sides of the number of blocks
(8192) from which the stride is 1024. Gradients against the oracle, or, in the larger images, against 8-pixel tiles,
whose walks are not cut."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_14244_gb300 import igs, scenes

from . import _gpu
from ._tiny import scene_from

pytestmark = pytest.mark.gpu


def _faint(n, seed, sigma=(0.05, 0.1), spread=0.5):
    """n faint Gaussians of which a pixel blends a few per cent (opacities just above 1/255: the
    core of each alone), so that no pixel stops and walks are as long as the lists."""
    rng = np.random.default_rng(seed)
    means = rng.uniform(-spread, spread, (n, 3))
    return scene_from(means, rng.uniform(*sigma, n), rng.uniform(0.0042, 0.006, n), rng.uniform(0, 1, (n, 3)))


def _check(sc, cam, tile):
    W = np.random.default_rng(3).normal(size=(3, cam.height, cam.width)).astype(np.float32)
    r, f, scene, _ = _gpu.run_forward(sc, cam, tile=tile)
    segs = igs.frame_walk_segments(f)
    d_ms, d_op, d_col = [t.cpu().numpy().astype(np.float64)
                         for t in r.run_backward(scene, cam, f, torch.from_numpy(W).cuda())]
    ref = oracle.backward(sc, cam, W.astype(np.float64), mode=1)
    _gpu.grad_close(d_ms[:, :3], ref["d_means"], "means")
    _gpu.grad_close(d_ms[:, 3], ref["d_sigma"], "sigma")
    _gpu.grad_close(d_op, ref["d_opac"], "opacity")
    _gpu.grad_close(d_col, ref["d_color"].reshape(d_col.shape), "color")
    return segs


def _check_uncut(sc, cam, tile):
    """The gradients with this tile size are those with 8-pixel tiles, whose walks are not cut. (The
    same FP32 decisions on both sides; so many entries at the edge of alpha_min leave the FP64 oracle
    a decision of its own here and there.)"""
    G = torch.from_numpy(np.random.default_rng(4).normal(size=(3, cam.height, cam.width)).astype(np.float32)).cuda()
    got = {}
    for t in (8, tile):
        r, f, scene, _ = _gpu.run_forward(sc, cam, tile=t)
        got[t] = [x.cpu().numpy().astype(np.float64) for x in r.run_backward(scene, cam, f, G)]
    for a, b, name in zip(got[tile], got[8], ("means and sigma", "opacity", "color")):
        _gpu.grad_close(a, b, name)
    return f


@pytest.mark.parametrize("n", [255, 256, 257, 511, 512, 513, 4095, 4097, 4353, 4609])
def test_around_the_stride(n):
    # wide enough that every Gaussian reaches the one tile: the list is n long
    sc = _faint(n, n, sigma=(0.25, 0.5))
    cam = scenes.pinhole((0.0, 0.0, -2.0), 16, 16, 16.0)
    segs = _check(sc, cam, 16)
    assert (segs > 0) == (n > 256)


def test_more_than_64_segments():
    # nearly 60,000 in the one tile's list: its four blocks share room for some 980 segments, of
    # which about half may be short ones, and a block takes one slot ahead; more than 64 each
    sc = _faint(60_000, 8, sigma=(0.1, 0.3))
    segs = _check(sc, scenes.pinhole((0.0, 0.0, -2.0), 16, 16, 16.0), 16)
    assert 4 * 130 < segs < 980


@pytest.mark.parametrize("n,w,h", [(20_000, 64, 48), (40_000, 64, 64)])
def test_lists_too_long_for_their_share_of_the_pool(n, w, h):
    # cut every 256 the lists would need more segments than there is room for; every 1024 they do not
    sc = _faint(n, 11, sigma=(0.1, 0.3))
    cam = scenes.pinhole((0.0, 0.0, -2.0), w, h, float(w))
    r, f, scene, _ = _gpu.run_forward(sc, cam, tile=16)
    rg = f.ranges().cpu().numpy().astype(np.int64)
    room = 16 * n // 1040 + 64 * (h // 16)  # the depth items' and the level-1 counts' bytes
    need = 4 * ((rg[:, 1] - rg[:, 0]) // 256 + 1).sum()
    assert 0 < igs.frame_walk_segments(f) < need and room < need
    _check_uncut(sc, cam, 16)


def test_first_blend_far_down_the_list():
    # the front 3000 lie over the left 8 columns of a 32-pixel tile, the rest over the right ones
    n = 6000
    sc = _faint(n, 9, sigma=(0.03, 0.06))
    rng = np.random.default_rng(10)
    z = np.sort(rng.uniform(-0.5, 0.5, n))
    u = np.where(np.arange(n) < 3000, rng.uniform(1.0, 7.0, n), rng.uniform(25.0, 31.0, n))
    sc.means_sigma[:, 0] = (u - 16.0) * (z + 2.0) / 32.0
    sc.means_sigma[:, 2] = z
    segs = _check(sc, scenes.pinhole((0.0, 0.0, -2.0), 32, 32, 32.0), 32)
    assert segs > 20


@pytest.mark.parametrize("side,n,sigma,cut", [
    (704, 10_000, (0.15, 0.25), True),    # 22 x 22 tiles of 16 blocks: cuts every 256
    (736, 10_000, (0.15, 0.25), False),   # 23 x 23 tiles, lists of 256 to 1024: every 1024, so none
    (736, 10_000, (0.4, 0.6), True),      # ... and lists of more
    (704, 1000, (0.3, 0.6), False), (736, 1000, (0.3, 0.6), False)])  # no room for segments at all
def test_either_side_of_few_blocks(side, n, sigma, cut):
    sc = _faint(n, side + n, sigma=sigma, spread=1.0)
    sc.means_sigma[:, 2] *= np.float32(0.25)
    cam = scenes.pinhole((0.0, 0.0, -2.0), side, side, 0.8 * side)
    f = _check_uncut(sc, cam, 32)
    rg = f.ranges().cpu().numpy().astype(np.int64)
    longest = (rg[:, 1] - rg[:, 0]).max()
    assert 256 < longest <= 1024 or sigma[0] > 0.2
    assert (igs.frame_walk_segments(f) > 0) == cut
