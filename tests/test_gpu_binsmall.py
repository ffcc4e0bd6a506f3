"""The binning of few Gaussians against the oracle's keys, at the edges of
its warps, sorted chunks, list rounds and its largest n, with ties, culled Gaussians and overflow."""
import numpy as np
import pytest

from paper_2403_14244_gb300 import igs, scenes

from . import _gpu
from .test_gpu_binning import _check_bitexact

pytestmark = pytest.mark.gpu

LARGEST = 65536  # the most Gaussians that take this route


def _scene(n, seed):
    sc = scenes.uniform_scene(n, seed)
    sc.means_sigma[::7, 2] = np.float32(0.25)     # many equal depths: ties by index
    sc.opacity[3::11] = np.float32(0.003)         # culled: below 1/255
    return sc


@pytest.mark.parametrize("tile", [8, 32])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 1023, 1025, 4095, 4096, 4097, 5119, 5120, 8193, 20000, LARGEST, LARGEST + 1])
def test_keys(n, tile):
    # 300 x 150: 38 tiles across at 8 pixels (more than one per warp), 10 at 32; both axes ragged
    _check_bitexact(_scene(n, n), scenes.pinhole((0.1, 0.2, -3.0), 300, 150, 200.0), tile)


def test_keys_wide_and_tall():
    sc = _scene(3000, 5)
    _check_bitexact(sc, scenes.pinhole((0.0, 0.0, -3.0), 16384, 16, 6000.0), 8)   # 2048 tiles across
    _check_bitexact(sc, scenes.pinhole((0.0, 0.0, -3.0), 16392, 16, 6000.0), 8)   # one more: the radix route
    _check_bitexact(_scene(9000, 6), scenes.pinhole((0.0, 0.0, -3.0), 200, 8, 90.0), 8)  # one row, many strips
    _check_bitexact(sc, scenes.pinhole((0.0, 0.0, -3.0), 24, 4096, 3000.0), 8)    # 512 rows


@pytest.mark.parametrize("n", [40, 5000])
def test_status_words_and_overflow(n):
    """A frame whose entries exceed its capacity reports them, aborts and binds nothing;
    the next frame of the right capacity is whole."""
    sc = _scene(n, 9)
    cam = scenes.pinhole((0.0, 0.0, -3.0), 200, 120, 150.0)
    r, f, scene, img = _gpu.run_forward(sc, cam, tile=16)
    st, info = igs.frame_status(f)
    words = f.info().cpu().numpy()
    assert st == igs.OK and words[3] == words[0] == words[5] and not words[8:].any()
    small = igs.Frame(n, int(info[0]) - 1, igs.camera(cam), r.opts)
    igs.project(scene, igs.camera(cam), r.opts, small)
    igs.bin_sort(small, r.opts)
    st, got = igs.frame_status(small)
    assert st == igs.ERR_CAPACITY and got[3] == info[0] and got[1] == info[1]
    exact = igs.Frame(n, int(info[0]), igs.camera(cam), r.opts)
    igs.project(scene, igs.camera(cam), r.opts, exact)
    igs.bin_sort(exact, r.opts)
    assert igs.frame_status(exact)[0] == igs.OK
    np.testing.assert_array_equal(exact.ranges().cpu().numpy(), f.ranges().cpu().numpy())
    np.testing.assert_array_equal(exact.vals(info[0]).cpu().numpy(), f.vals(info[0]).cpu().numpy())
