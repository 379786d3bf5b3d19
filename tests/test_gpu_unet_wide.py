"""The warm-start network's convolutions of many channels (64 output channels
a block, 16 input channels at a time), layer by layer as in
test_gpu_unet_shapes.py: channel counts that end inside a block and inside a
step, pixels of 8, 2 and 1 aligned channels, images that end inside a tile, and
the tiles of 16 x 16 pixels that large images take."""
import pytest

import test_gpu_unet_shapes as shapes
from test_gpu_unet import ms  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,width,H,W", [(2, 136, 80, 72), (2, 250, 8, 24), (2, 233, 16, 8),
                                              (2, 72, 216, 216), (2, 66, 216, 232),
                                              (2, 97, 208, 208)])
def test_each_wide_layer(ms, levels, width, H, W):  # noqa: F811
    shapes.test_each_layer(ms, levels, width, H, W)
