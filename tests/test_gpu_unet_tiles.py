"""The convolution tiles of the warm-start network at grids where they can go
wrong: several tiles along x (more than 126 voxels), tiles cut off by every
side of the grid, one tile for the whole grid, long thin grids.  Every layer
is held to the same bounds against the fp64 reference as on the small grids.
"""
import pytest

from . import test_gpu_unet as U

pytestmark = pytest.mark.gpu

FORWARD = [(8, 12, 132), (8, 8, 260), (12, 44, 128), (36, 8, 8), (20, 28, 52)]
BACKWARD = [(8, 12, 132), (20, 16, 28)]


@pytest.mark.parametrize("shape", FORWARD, ids=lambda s: "x".join(map(str, s)))
def test_forward_layers_on_every_kind_of_tile(shape):
    U.test_forward_layers_match_the_reference(shape)


@pytest.mark.parametrize("shape", BACKWARD, ids=lambda s: "x".join(map(str, s)))
def test_backward_layers_on_every_kind_of_tile(shape):
    U.test_backward_layers_match_the_reference(shape)
