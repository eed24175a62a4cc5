"""Wide layers on the halo kernel: one halo buffer and a ring of two or three
stages of weights, by TMA (blocks of 64 channels) and by pieces (48), one and
several tiles a block and tiles of output channels.  The check is that of
test_gpu_conv_halo.py: element by element against the oracle with the same
BF16 operand rounding, within the FP32 summation bound."""
import pytest

import test_gpu_conv_halo as H

pytestmark = pytest.mark.gpu

env = H.env


@pytest.mark.parametrize("shape", [(1, 32, 24, 384, 256), (1, 160, 136, 384, 192), (1, 32, 24, 320, 240), (1, 32, 24, 432, 256),
                                   (1, 16, 8, 448, 160), (2, 16, 24, 512, 64), (1, 32, 24, 384, 512)])
def test_wide_forward_layers(env, shape):
    assert env[2].nn_conv3x3_form(shape[1], shape[2], shape[3], shape[4]) == 2
    H.test_forward_branches(env, shape)
