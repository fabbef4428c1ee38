"""The convolution's strips of 128 columns and of whole rows, each with the tile
and block counts that choose them (comparison and bounds of
test_gpu_conv_sizes)."""
import pytest
from test_gpu_conv_sizes import test_convolution_and_gradients as check

pytestmark = pytest.mark.gpu

SIZES = [  # n, ci, co, h, w
    (1, 64, 192, 32, 128), (4, 64, 192, 32, 128), (20, 64, 192, 32, 128),  # blocks of 64: one, three, three with two tiles
    (16, 96, 32, 64, 256), (24, 32, 32, 32, 384),                          # four tiles: rows of 256, strips of 192
    (8, 96, 32, 64, 256), (3, 32, 32, 12, 640), (2, 32, 96, 8, 384), (1, 16, 128, 4, 512),
]


@pytest.mark.parametrize("n,ci,co,h,w", SIZES)
def test_strips(n, ci, co, h, w):
    check(n, ci, co, h, w)
