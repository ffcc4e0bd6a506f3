"""Frames of medium size, bit for bit against the oracle's keys: at the Gaussian counts where
the depth sort's blocks change (778 240 and one more) and where the chunks of the two walks
stop being shortened, in a frame whose capacity is exactly its entries (the level-2 chunks then
have the least room) and in a roomy one; then a frame with too little capacity."""
import numpy as np
import pytest

from paper_2403_14244_gb300 import igs, scenes

from . import _gpu
from .test_gpu_binning import _check_bitexact

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [65537, 151_003, 778_240, 778_241])
def test_keys(n):
    sc = scenes.clustered_scene(n, 31)
    sc.opacity[5::9] = np.float32(0.002)          # culled: below 1/255
    _check_bitexact(sc, scenes.pinhole((0.2, 0.1, -3.0), 333, 217, 180.0), 16)


@pytest.mark.parametrize("size", [(333, 217, 16), (1280, 720, 8), (64, 1100, 8), (40, 40, 32)])
@pytest.mark.parametrize("n", [65537, 200_003])
def test_exact_capacity(n, size):
    w, h, tile = size
    sc = scenes.clustered_scene(n, 32)
    cam = scenes.pinhole((0.0, 0.0, -3.0), w, h, 0.6 * max(w, h))
    r, f, scene, img = _gpu.run_forward(sc, cam, tile=tile)
    st, info = igs.frame_status(f)
    assert st == igs.OK
    for room, want in ((0, igs.OK), (1, igs.OK), (-1, igs.ERR_CAPACITY)):
        g = igs.Frame(n, int(info[0]) + room, igs.camera(cam), r.opts)
        igs.project(scene, igs.camera(cam), r.opts, g)
        igs.bin_sort(g, r.opts)
        st, got = igs.frame_status(g)
        assert st == want and got[3] == info[0] and got[1] == info[1]
        if want == igs.OK:
            np.testing.assert_array_equal(g.ranges().cpu().numpy(), f.ranges().cpu().numpy())
            np.testing.assert_array_equal(g.vals(info[0]).cpu().numpy(), f.vals(info[0]).cpu().numpy())
