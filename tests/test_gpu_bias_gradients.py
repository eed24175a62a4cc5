"""Bias and head gradients of the surrogate network: they repeat bit for bit
from call to call (partial sums added in an order that the sizes give), and
they are the right sums.

For the second part all weights, biases, inputs and output gradients are
positive, so that every ReLU is open and every sum has terms of one sign, and
output channel 0 of each convolution is held at 1 (weights 0, bias 1).  A
weight gradient against an input channel that is 1 everywhere is then the sum
of the layer's output gradient, the bias gradient itself, up to the rounding of
its terms to BF16 (2^-9 relative) and the FP32 sums (P 2^-24 each)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# levels, base, batch, H, W: the most blocks a layer takes, single blocks at the
# deepest level, the widest layers, the narrowest partial rows
ARCHS = [(3, 16, 8, 128, 128), (3, 16, 1, 32, 32), (2, 64, 1, 16, 48), (3, 64, 1, 64, 32), (5, 16, 1, 128, 128)]


@pytest.fixture(scope="module")
def env():
    import torch

    from oracle import unet_oracle as U
    from paper_1606_09432_gb300 import build as B
    from paper_1606_09432_gb300 import lbpf as L
    B.build()
    return torch, U, L


def slices(U, levels, base):
    """Per convolution (cin, cout, weights, bias), then the head's."""
    off, out = 0, []
    for ci, co in U.layers((levels, base)):
        n = 9 * ci * co
        out.append((ci, co, slice(off, off + n), slice(off + n, off + n + co)))
        off += n + co
    return out, slice(off, off + 2 * base), slice(off + 2 * base, off + 2 * base + 2)


@pytest.mark.parametrize("levels,base,batch,H,W", ARCHS)
def test_bias_and_head_gradients_repeat(env, levels, base, batch, H, W):
    torch, U, L = env
    net = L.Net(H, W, batch=batch, seed=3, levels=levels, base=base)
    convs, hw, hb = slices(U, levels, base)
    torch.manual_seed(levels)
    x = torch.randn(batch, H, W, 5, device="cuda")
    dy = torch.randn(batch, H, W, 2, device="cuda")
    keep = np.r_[tuple(c[3] for c in convs) + (hw, hb)]
    net.forward(x)
    first = net.backward(dy)[keep]
    assert np.any(first != 0)
    for _ in range(5):
        net.forward(x)
        assert np.array_equal(net.backward(dy)[keep], first)


@pytest.mark.parametrize("levels,base,batch,H,W", ARCHS)
def test_bias_gradients_are_the_sums(env, levels, base, batch, H, W):
    torch, U, L = env
    net = L.Net(H, W, batch=batch, seed=3, levels=levels, base=base)
    convs, hw, hb = slices(U, levels, base)
    rng = np.random.default_rng(levels * base)
    p = np.zeros(net.n_params, np.float32)
    for ci, co, sw, sb in convs:
        w = rng.uniform(0.5, 1.5, (9, co, ci)) / (9 * ci)
        w[:, 0, :] = 0.0
        p[sw] = w.ravel()
        p[sb] = rng.uniform(0.5, 1.0, co)
        p[sb][0] = 1.0
    p[hw] = rng.uniform(0.5, 1.0, 2 * base)
    net.set_params(p)
    x = rng.uniform(0.1, 0.9, (batch, H, W, 5)).astype(np.float32)
    x[..., 4] = 1.0
    dy = rng.uniform(0.5, 1.5, (batch, H, W, 2)).astype(np.float32)
    net.forward(torch.from_numpy(x).cuda())
    g = net.backward(torch.from_numpy(dy).cuda()).astype(np.float64)
    P = batch * H * W
    sums = 2.0 * P * 2.0 ** -24
    ph = x[..., 0].astype(np.float64)
    want = np.array([(dy[..., 0] * (1 - ph * ph)).sum(), dy[..., 1].sum(dtype=np.float64)])
    assert np.all(np.abs(g[hb] - want) <= (sums + 2.0 ** -21) * want)  # the gate's three roundings
    assert np.all(np.abs(g[hw].reshape(2, base)[:, 0] - want) <= (sums + 2.0 ** -21) * want)
    for k, (ci, co, sw, sb) in enumerate(convs):
        one = g[sw].reshape(9, co, ci)[:, :, 4 if k == 0 else 0]  # the input channel that is 1
        db = g[sb]
        assert np.all(db > 0)
        assert np.all(np.abs(one - db) <= (2.0 ** -9 + 2 * sums) * db), k
