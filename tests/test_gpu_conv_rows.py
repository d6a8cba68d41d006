"""The two-row pixel tiles of the convolutions against the FP64 oracle.

A convolution takes two image rows per tile where one-row tiles would number
at least 304 (ceil(W / 128) x H) and the level is at least 128 wide: at
400 x 304 that is so at level 0 (1216 tiles) and level 1 (304 tiles, the
threshold itself), both with a ragged last tile (400 = 3 x 128 + 16,
200 = 128 + 72); at 384 x 112 at level 0 only, with full tiles.  The bounds
are those of the layer-by-layer comparison, which covers the one-row tiles."""
import pytest

import test_gpu_cnn_layers as layers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W, H", [(400, 304), (384, 112)])
def test_two_row_tiles_in_lockstep(mvs_lib, W, H):
    layers.test_every_layer_in_lockstep(mvs_lib, W, H)
