"""Convolutions of images whose halo offsets do not fit in 32 bits (rows of more
than 2^27 floats): the same bits as on a crop, for the forward kernel and for
the weight gradient of an output gradient that is zero outside the crop."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,cin", [(2 ** 19, 256), (2 ** 20 + 8, 128)])
def test_rows_of_more_than_2_27_floats(W, cin):
    import torch

    from paper_1606_09432_gb300 import lbpf as L
    H, cout, x0, w = 48, 16, W - 4096, 64
    if torch.cuda.mem_get_info()[0] < 40e9:
        pytest.skip("needs 32 GB of device memory")
    g = torch.Generator(device="cuda").manual_seed(W)
    x = torch.zeros((1, H, W, cin), device="cuda")
    x[:, :, x0 - 8:x0 + w + 8] = torch.randn((1, H, w + 16, cin), device="cuda", generator=g)
    crop = x[:, :, x0 - 8:x0 + w + 8].contiguous()
    wt = (torch.randn((9, cout, cin), device="cuda", generator=g) / 48).to(torch.bfloat16)
    b = torch.randn(cout, device="cuda", generator=g)
    y = torch.full((1, H, W, cout), float("nan"), device="cuda")
    yc = torch.empty((1, H, w + 16, cout), device="cuda")
    L.nn_conv3x3(x, wt, b, y)
    L.nn_conv3x3(crop, wt, b, yc)
    torch.cuda.synchronize()
    assert torch.equal(y[:, :, x0:x0 + w], yc[:, :, 8:8 + w])
    assert torch.equal(y[:, :, 16:x0 - 16], b.expand(1, H, x0 - 32, cout))
    # weight gradient: one non-zero tile of dy, so that its sums have one block's order
    y.zero_()
    yc.zero_()
    y[:, 16:32, x0:x0 + 8] = torch.randn((1, 16, 8, cout), device="cuda", generator=g)
    yc[:, 16:32, 8:16] = y[:, 16:32, x0:x0 + 8]
    dw, dwc = (torch.zeros((9, cout, cin), device="cuda") for _ in range(2))
    L.nn_conv3x3_wgrad(x, y, dw)
    L.nn_conv3x3_wgrad(crop, yc, dwc)
    torch.cuda.synchronize()
    assert L.nn_conv_error() == 0
    assert torch.equal(dw, dwc) and torch.any(dw != 0)
