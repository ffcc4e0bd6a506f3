"""The lines between the binning of few Gaussians and the general route, in Gaussians and in
Gaussians times tiles: on either side a frame's keys match the oracle's, and the launches show
which route it took."""
import pytest

from paper_2403_14244_gb300 import igs, scenes

from . import _gpu
from .test_gpu_binning import _check_bitexact

pytestmark = pytest.mark.gpu


def _launches(sc, cam, tile):
    """Kernels of one igs_bin_sort."""
    r, f, scene, img = _gpu.run_forward(sc, cam, tile=tile)
    before = igs.launch_count()
    igs.bin_sort(f, r.opts)
    return igs.launch_count() - before


@pytest.mark.parametrize("n,w,h,tile,small", [
    (49152, 300, 150, 16, True), (49153, 300, 150, 16, False),
    # 2048 x 64 tiles: 16384 Gaussians make 2^31 of them, one more is past the line
    (16384, 16384, 512, 8, True), (16385, 16384, 512, 8, False),
    # as few Gaussians as in an ordinary small frame, on more tiles than one has
    (24576, 3840, 2160, 8, False), (32768, 4096, 2160, 8, False), (32768, 3840, 2160, 16, True)])
def test_line(n, w, h, tile, small):
    sc = scenes.uniform_scene(n, n % 97)
    sc.means_sigma[::5, 2] = sc.means_sigma[0, 2]  # ties in depth
    sc.means_sigma[:, 3] *= 0.5
    cam = scenes.pinhole((0.1, 0.2, -3.0), w, h, 0.6 * w)
    assert _check_bitexact(sc, cam, tile) > n // 4
    assert (_launches(sc, cam, tile) <= 3) == small
