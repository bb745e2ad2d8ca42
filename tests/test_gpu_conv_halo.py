"""The halo-tile convolution (images narrower than 48 pixels, tiles of 8 x 16)
at the sizes where it can go wrong: one pixel, one less and one more than a
tile in each direction, the widest image it takes and the first one it leaves,
the most input channels that fit its shared memory and more (another kernel),
output channels split over several CTAs or not; BF16 and E4M3.  Checked as the
other single layers are: against the float64 convolution of the same values."""
import pytest

from tests.test_gpu_denoise import test_conv3x3_e4m3_layer_matches_library as check_e4m3
from tests.test_gpu_denoise import test_conv3x3_layer_matches_library as check_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,H,W", [(16, 16, 1, 1), (16, 32, 15, 7), (32, 48, 17, 9), (48, 96, 16, 8), (64, 64, 33, 47),
                                          (64, 64, 33, 48), (96, 256, 5, 31), (176, 112, 18, 10), (608, 16, 16, 9),
                                          (624, 16, 16, 9), (1024, 32, 3, 20), (32, 32, 200, 40)])
def test_bf16_layer(cuda_lib, cin, cout, H, W):
    check_bf16(cuda_lib, cin, cout, H, W, True)


@pytest.mark.parametrize("cin,cout,H,W", [(32, 16, 1, 1), (64, 48, 17, 9), (160, 64, 33, 47), (1216, 16, 16, 9),
                                          (1248, 16, 16, 9)])
def test_e4m3_layer(cuda_lib, cin, cout, H, W):
    check_e4m3(cuda_lib, cin, cout, H, W, False)
