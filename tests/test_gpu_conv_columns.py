"""Column-walking convolutions whose columns of tiles end within CTAs' runs, on more
than four tiles per SM (fewer take the other kernel), against FP64 as in
test_gpu_conv_roll.py."""
import pytest
import test_gpu_conv_roll as roll

pytestmark = pytest.mark.gpu


# six columns; two input rows a stage (64 channels) and one (128), ragged N
@pytest.mark.parametrize("B,H,width,C,N", [(3, 120, 256, 64, 64), (3, 110, 256, 128, 64), (2, 110, 384, 128, 40),
                                           (1, 207, 384, 64, 24), (7, 53, 256, 32, 32)])
@pytest.mark.parametrize("fp32", [0, 1])
def test_outputs_match_fp64(B, H, width, C, N, fp32):
    roll.test_outputs_match_fp64(B, H, width, C, N, fp32)
