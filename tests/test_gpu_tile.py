"""The one-tile step of small 2D domains against the marching step kernel
(LBPF_KERNEL=generic).  Both evaluate the same operations in the same order:
fields, populations and the index must agree bit for bit, for every storage
form, with walls, several crystals and both gradients, at the edges of the
tile (30 x 6 sites) and down to the smallest domains."""
import numpy as np
import pytest

from helpers import gpu_run
from paper_1606_09432_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1606_09432_gb300 import build as B
    from paper_1606_09432_gb300 import lbpf
    B.build()
    lbpf.load()
    return lbpf


def smooth_fields(shape, seed, dtype):
    rng = np.random.default_rng(seed)
    waves = [np.cos(2 * np.pi * (np.arange(n) / n + rng.random())) for n in shape]
    w = waves[0][:, None, None] + waves[1][None, :, None] + waves[2][None, None, :]
    phi = np.tanh(w - w[:1, :1, :1]) + 0.01 * rng.standard_normal(shape)
    return phi.astype(dtype), (-0.3 + 0.05 * w + 0.01 * rng.standard_normal(shape)).astype(dtype)


def compare(L, monkeypatch, shape, precision, crystals, steps=(1, 1, 2, 19), **kw):
    fields = smooth_fields(shape, sum(shape) + precision, np.float64 if precision == 0 else np.float32)
    runs = []
    for kernel in ("", "generic"):
        monkeypatch.setenv("LBPF_KERNEL", kernel)
        runs.append(gpu_run(L, 0, shape, W.C1_PARAMS, crystals, fields=fields, precision=precision, **kw))
    a, b = runs
    for k in steps:
        for s in runs:
            s.step(k)
        if k != 1:
            for x, y in zip(a.fields(), b.fields()):
                assert np.array_equal(x, y)
    for which in (0, 1):
        assert np.array_equal(a.populations(which), b.populations(which))
    if len(crystals) > 1:
        assert np.array_equal(a.field(L.LBPF_FIELD_INDEX), b.field(L.LBPF_FIELD_INDEX))


@pytest.mark.parametrize("precision", range(5))
@pytest.mark.parametrize("shape", [(1, 2, 2), (1, 3, 5), (1, 6, 30), (1, 7, 31), (1, 13, 29), (1, 12, 91), (1, 64, 128)])
def test_tile_step_matches_march(L, monkeypatch, shape, precision):
    compare(L, monkeypatch, shape, precision, [dict(kind=0, eps=0.05)])


@pytest.mark.parametrize("bc,grad", [(1, 0), (2, 0), (3, 0), (3, 1), (0, 1)])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_tile_step_walls_and_gradients(L, monkeypatch, bc, grad, precision):
    compare(L, monkeypatch, (1, 25, 61), precision, [dict(kind=1, eps=0.05, q=6)], bc=bc, grad=grad)


@pytest.mark.parametrize("precision", [0, 1, 4])
def test_tile_step_crystal_index(L, monkeypatch, precision):
    """Three seeds: the index field spreads over the tiles' edges."""
    shape = (1, 40, 95)
    cr = [dict(kind=1, eps=0.05, q=4, phi0=0.3 * k) for k in range(3)]
    seeds = [(28.0, 5.0, 0.0, 4.0, 0), (60.0, 20.0, 0.0, 5.0, 1), (10.0, 33.0, 0.0, 4.0, 2)]
    out = []
    for kernel in ("", "generic"):
        monkeypatch.setenv("LBPF_KERNEL", kernel)
        s = gpu_run(L, 0, shape, W.C1_PARAMS, cr, seeds=seeds, precision=precision, xi=0.1)
        s.step(60)
        out.append(s.fields() + (s.field(L.LBPF_FIELD_INDEX),))
    for x, y in zip(*out):
        assert np.array_equal(x, y)
    assert len(np.unique(out[0][2])) == 4


def test_set_schedule_returns_to_the_march(L, monkeypatch):
    monkeypatch.setenv("LBPF_KERNEL", "")
    fields = smooth_fields((1, 33, 70), 1, np.float32)
    a = gpu_run(L, 0, (1, 33, 70), W.C1_PARAMS, [dict(kind=0, eps=0.05)], fields=fields, precision=1)
    b = gpu_run(L, 0, (1, 33, 70), W.C1_PARAMS, [dict(kind=0, eps=0.05)], fields=fields, precision=1)
    a.step(20)
    L.lbpf_set_schedule(a.ctx, 16, 5)
    assert a.query(L.LBPF_Q_SEGMENT) == 5
    a.step(20)
    b.step(40)
    for x, y in zip(a.fields(), b.fields()):
        assert np.array_equal(x, y)
