"""The tensor-core weight gradients of the warm-start network at grids whose
levels end in partial voxel tiles: 16^3 (4096, 512, 64, 8 voxels), 24^3
(13824, 1728, 216, 27: remainders of the 64-voxel tile and of the voxel
chunks, odd coarsest grid).  Held to the bounds of the forward and gradient
parity test."""

import pytest

from test_gpu_unet import test_forward_and_gradients_match_oracle as forward_and_gradients_match_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 24])
def test_weight_gradients_at_partial_tiles(n):
    forward_and_gradients_match_oracle(n)
