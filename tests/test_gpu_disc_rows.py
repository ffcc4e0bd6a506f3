"""Disc footprints (footprint 1) of Gaussians whose centres lie beside the image, bit for bit
against the oracle's keys: their rectangles span tile rows in which the disc misses the grid,
so that the rows of the rectangles outnumber the entries. On both ways of the tile ranges
(few and many tiles), in a frame of default capacity and in one that holds exactly its entries,
and as the image of rectangle footprints."""
import numpy as np
import pytest

import oracle
from paper_2403_14244_gb300 import igs, scenes

from . import _gpu
from .test_gpu_binning import _check_bitexact

gpu = pytest.mark.gpu


def _beside(n, side, w, h, among=0):
    """n discs of radius about 200 px whose centres lie 196 px beside the image of the camera,
    at half its height, and `among` ordinary Gaussians. side: -1 left, 1 right, 0 both."""
    cam = scenes.pinhole((0.0, 0.0, -4.0), w, h, 400.0)
    rng = np.random.default_rng(n + side)
    sc = scenes.uniform_scene(n + among, 17)
    at = np.where(rng.random(n) < 0.5, -1, 1) if side == 0 else np.full(n, side)
    u = np.where(at < 0, -196.0, w + 196.0) + rng.uniform(-1.0, 1.0, n)
    v = 0.5 * h + rng.uniform(-2.0, 2.0, n)
    z = rng.uniform(4.0, 4.2, n)
    sc.means_sigma[:n] = np.stack([(u - cam.cx) * z / 400.0, (v - cam.cy) * z / 400.0, z - 4.0,
                                   200.0 / 3.297 * z / 400.0], 1)  # radius = 3.297 s at opacity 0.9
    sc.opacity[:n] = np.float32(0.9)
    order = rng.permutation(n + among)
    sc.means_sigma[:], sc.opacity[:], sc.color[:] = sc.means_sigma[order], sc.opacity[order], sc.color[order]
    return sc, cam


CASES = [(2000, -1, 640, 480, 8, 0), (2000, 1, 640, 480, 8, 0), (900, 0, 1280, 960, 8, 0), (4000, 0, 640, 480, 16, 3000),
         (40, -1, 640, 480, 8, 0), (70_000, 1, 333, 480, 32, 5000)]


@pytest.mark.parametrize("case", CASES)
def test_rows_outnumber_entries(case):
    """The scenes below are what they say: more (Gaussian, row) pairs in the rectangles than entries,
    and in the rows a disc touches, which are consecutive, never more than entries."""
    n, side, w, h, tile, among = case
    sc, cam = _beside(n, side, w, h, among)
    p = oracle.project(sc.means_sigma, sc.opacity, cam, tile, 1)
    kept = np.nonzero(p["count"] > 0)[0]
    assert len(kept) >= 0.9 * n
    rows = touched = 0
    for i in kept:
        x0, y0, x1, y1 = p["rect"][i]
        xa, xb = oracle.row_span(p["u"][i], p["v"][i], p["r"][i], np.arange(y0, y1 + 1), x0, x1, tile)
        on = np.nonzero(xa <= xb)[0]
        assert on.size and on[-1] - on[0] + 1 == on.size
        rows += y1 - y0 + 1
        touched += on.size
    assert touched <= p["count"].sum()
    if among == 0:
        assert rows > p["count"].sum()


@gpu
@pytest.mark.parametrize("case", CASES)
def test_keys(case):
    n, side, w, h, tile, among = case
    sc, cam = _beside(n, side, w, h, among)
    m = _check_bitexact(sc, cam, tile, 1)
    r, f, scene, img = _gpu.run_forward(sc, cam, tile=tile, footprint=1)
    _, _, _, img0 = _gpu.run_forward(sc, cam, tile=tile, footprint=0)
    np.testing.assert_array_equal(img, img0)
    for room, want in ((0, igs.OK), (-1, igs.ERR_CAPACITY)):
        g = igs.Frame(scene.n, m + room, igs.camera(cam), r.opts)
        igs.project(scene, igs.camera(cam), r.opts, g)
        igs.bin_sort(g, r.opts)
        st, got = igs.frame_status(g)
        assert st == want and got[3] == m
        if want == igs.OK:
            np.testing.assert_array_equal(g.ranges().cpu().numpy(), f.ranges().cpu().numpy())
            np.testing.assert_array_equal(g.vals(m).cpu().numpy(), f.vals(m).cpu().numpy())
