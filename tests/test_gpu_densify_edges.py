"""Densify / prune of 3D Gaussians at the edges of a block's 512 Gaussians, with room for every
division, for some and for none, rows copied as float4 and as floats: bit for bit against the
oracle."""
import pytest

from tests import test_gpu_densify3d as base

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sh,mode", [(-1, 0), (3, 1)])
@pytest.mark.parametrize("n", [255, 257, 511, 512, 513, 1023, 1025])
@pytest.mark.parametrize("room", [0, 100, 10_000])
def test_block_edges(n, room, sh, mode):
    base.test_densify_bit_exact(n, n + room, sh, mode)
