"""Branches of the halo convolutions that depend on sizes: several tiles a
block (persistent loop, every number of halo buffers), resident weights with
an unrolled or a general channel count, weights streamed through the ring
(blocks of 64, 48 and 16 channels, one and two halo buffers), and the weight
gradient with nine and with three taps a block, several channel tiles and
unaligned inputs.  Against the oracle with the same BF16 operand rounding,
element by element within the FP32 summation bound gamma_K of the absolute
terms (K terms, u = 2^-24), as in test_gpu_conv.py."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U24 = 2.0 ** -24


@pytest.fixture(scope="module")
def env():
    import torch

    from oracle import unet_oracle as U
    from paper_1606_09432_gb300 import build as B
    from paper_1606_09432_gb300 import lbpf as L
    B.build()
    L.load()
    return torch, U, L


@pytest.mark.parametrize("shape", [(1, 256, 320, 16, 16), (2, 96, 216, 32, 16), (1, 64, 40, 176, 16), (1, 64, 48, 96, 256),
                                   (1, 32, 24, 176, 256), (2, 32, 168, 64, 128), (1, 32, 24, 384, 32)])
def test_forward_branches(env, shape):
    torch, U, L = env
    n, H, W, cin, cout = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((n, H, W, cin)).astype(np.float32)
    wq = U.bf16(rng.standard_normal((9, cout, cin)) / np.sqrt(9 * cin))
    b = rng.standard_normal(cout).astype(np.float32)
    y = torch.full((n, H, W, cout), float("nan"), device="cuda")
    L.nn_conv3x3(torch.from_numpy(x).cuda(), torch.from_numpy(wq.astype(np.float32)).cuda().to(torch.bfloat16),
                 torch.from_numpy(b).cuda(), y, relu=True)
    torch.cuda.synchronize()
    assert L.nn_conv_error() == 0
    x, b = x.astype(np.float64), b.astype(np.float64)
    want = np.maximum(U.conv3x3(x, wq, b, emulate=True), 0.0)
    K = 9 * cin + 1
    bar = K * U24 / (1 - K * U24) * (U.conv3x3(np.abs(U.bf16(x)), np.abs(wq)) + np.abs(b))
    assert np.all(np.abs(y.cpu().numpy() - want) <= bar + 1e-30)


@pytest.mark.parametrize("shape,shift", [((1, 256, 320, 16, 32), 0), ((1, 96, 216, 48, 16), 0), ((1, 32, 24, 176, 144), 0),
                                         ((1, 64, 40, 192, 272), 0), ((2, 32, 24, 32, 32), 1)])
def test_weight_gradient_branches(env, shape, shift):
    """shift: floats by which x, dy and dw are off a 16-byte boundary."""
    torch, U, L = env
    n, H, W, cin, cout = shape
    rng = np.random.default_rng(sum(shape) + shift)

    def dev(a):
        t = torch.empty(a.size + shift, device="cuda")
        t[shift:] = torch.from_numpy(a.astype(np.float32).ravel()).cuda()
        return t[shift:].view(a.shape)

    x, dy = rng.standard_normal((n, H, W, cin)), rng.standard_normal((n, H, W, cout))
    d0 = rng.standard_normal((9, cout, cin)).astype(np.float32)
    dw = dev(d0)
    L.nn_conv3x3_wgrad(dev(x), dev(dy), dw)
    torch.cuda.synchronize()
    assert L.nn_conv_error() == 0
    x, dy = x.astype(np.float32).astype(np.float64), dy.astype(np.float32).astype(np.float64)
    want = d0.astype(np.float64) + U.conv3x3_wgrad(x, dy, emulate=True)
    K = n * H * W + 1
    bar = K * U24 / (1 - K * U24) * (np.abs(d0) + U.conv3x3_wgrad(np.abs(x), np.abs(dy), emulate=True))
    assert np.all(np.abs(dw.cpu().numpy().astype(np.float64) - want) <= bar)
