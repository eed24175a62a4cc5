"""Which kernel a convolution layer takes (host arithmetic, no GPU call): on
images of whole 16 x 8 tiles every layer whose halo and two stages of weights
fit in shared memory takes the halo kernel, the wide ones among them."""
import pytest


@pytest.fixture(scope="module")
def L():
    from paper_1606_09432_gb300 import build as B
    from paper_1606_09432_gb300 import lbpf
    B.build()
    return lbpf


@pytest.mark.parametrize("cin,cout", [(384, 256), (384, 192), (320, 256), (448, 128), (448, 160), (512, 64), (512, 80),
                                      (432, 256), (384, 384), (384, 512), (320, 768)])
def test_wide_layers_take_the_halo_kernel(L, cin, cout):
    assert L.nn_conv3x3_form(64, 64, cin, cout) == 2


def test_every_layer_that_two_stages_hold_takes_the_halo_kernel(L):
    for cin in range(16, 769, 16):
        kc = cin if cin <= 64 else next(k for k in (64, 48, 32, 16) if cin % k == 0)
        for cout in range(16, 769, 16):
            tiles = (cout + 255) // 256
            if cout % (16 * tiles):
                continue
            if 2 * 180 * cin + 4 * kc * cout // tiles <= 200 * 1024:
                assert L.nn_conv3x3_form(16, 8, cin, cout) > 0, (cin, cout)


def test_forms_of_other_layers(L):
    assert L.nn_conv3x3_form(64, 64, 32, 32) == 1
    assert L.nn_conv3x3_form(64, 60, 32, 32) == L.nn_conv3x3_form(63, 64, 32, 32) == 0
    assert L.nn_conv3x3_form(64, 64, 768, 256) == 0
    for bad in ((64, 64, 8, 16), (64, 64, 24, 16), (64, 64, 16, 272), (0, 64, 16, 16)):
        with pytest.raises(L.LbpfError):
            L.nn_conv3x3_form(*bad)
