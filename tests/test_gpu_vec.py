"""The vector step (two launches, four sites a thread; 3D, 16-bit deviations)
against the one-launch step kernel (LBPF_KERNEL=vector and generic).

Both evaluate the same operations in the same order, so the fields and the
populations must agree bit for bit.  Sizes sit at the edges of the vector
form's tile (64 x 12 sites, rows padded to whole vectors of four): the
smallest rows, one and several segments with short last ones of every length
modulo four, rows of blocks
that end inside the domain, and columns of two planes.  Reads between the
steps put the heat state through both of its forms (synchronised, lagged)."""
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


SHAPES = [(2, 2, 8), (2, 3, 9), (4, 13, 66), (5, 14, 67), (6, 12, 127), (3, 25, 197), (3, 13, 12), (5, 12, 64), (4, 25, 72), (7, 11, 128), (9, 37, 140), (40, 24, 200)]
FORM = dict(kind=3, eps=0.02, gamma=-0.02)


def smooth_fields(shape, seed):
    """A wavy interface with a little noise."""
    rng = np.random.default_rng(seed)
    waves = [np.cos(2 * np.pi * (np.arange(n) / n + rng.random())) for n in shape]
    w = waves[0][:, None, None] + waves[1][None, :, None] + waves[2][None, None, :]
    phi = np.tanh(w) + 0.01 * rng.standard_normal(shape)
    u = -0.4 + 0.05 * w + 0.01 * rng.standard_normal(shape)
    return phi.astype(np.float32), u.astype(np.float32)


def both(L, monkeypatch, make):
    out = []
    for kernel in ("vector", "generic"):
        monkeypatch.setenv("LBPF_KERNEL", kernel)
        out.append(make())
    return out


@pytest.mark.parametrize("precision", [2, 3, 4])
@pytest.mark.parametrize("lattice", [1, 2, 3])
@pytest.mark.parametrize("shape", SHAPES)
def test_vector_step_matches_one_launch_step(L, monkeypatch, shape, lattice, precision):
    prm = dict(W.C3D_PARAMS, delta=0.4)
    phi, u = smooth_fields(shape, sum(shape) + lattice)
    a, b = both(L, monkeypatch, lambda: gpu_run(L, lattice, shape, prm, [FORM], fields=(phi, u), precision=precision))
    for steps in (1, 1, 2, 21):
        for s in (a, b):
            s.step(steps)
        if steps != 1:
            for x, y in zip(a.fields(), b.fields()):
                assert np.array_equal(x, y)
    for which in (0, 1):
        assert np.array_equal(a.populations(which), b.populations(which))


@pytest.mark.parametrize("bc", [1, 2, 4, 7])
@pytest.mark.parametrize("lattice,grad,nx", [(1, 0, 76), (2, 0, 76), (3, 0, 77), (1, 1, 74), (1, 0, 67), (2, 0, 65)])
def test_vector_step_walls_and_gradients(L, monkeypatch, bc, lattice, grad, nx):
    shape = (9, 14, nx)
    prm = dict(W.C3D_PARAMS, delta=0.4)
    phi, u = smooth_fields(shape, bc + 10 * lattice + grad)
    a, b = both(L, monkeypatch, lambda: gpu_run(L, lattice, shape, prm, [FORM], fields=(phi, u), precision=2, bc=bc,
                                                grad=grad))
    for s in (a, b):
        s.step(17)
    for x, y in zip(a.fields(), b.fields()):
        assert np.array_equal(x, y)


def test_padded_rows_through_every_read(L, monkeypatch):
    """Rows of 67 sites padded to 68: measurement, tip radius, a_s and the
    seeded start against the one-launch kernel's dense arrays."""
    prm = dict(W.C3D_PARAMS, delta=0.4)
    a, b = both(L, monkeypatch, lambda: gpu_run(L, 1, (40, 37, 67), prm, [FORM], seeds=[(33.0, 18.0, 20.0, 8.0, 0)],
                                                precision=2))
    for s in (a, b):
        s.step(12)
    ma, mb = a.measure(33, 18, 20), b.measure(33, 18, 20)
    assert np.array_equal(ma[0], mb[0]) and ma[1] == mb[1] and ma[2] == mb[2]
    assert a.tip_radius(33, 18, 20, 0) == b.tip_radius(33, 18, 20, 0)
    assert np.array_equal(a.anisotropy_field(), b.anisotropy_field())
    assert np.array_equal(a.field(L.LBPF_FIELD_INDEX), b.field(L.LBPF_FIELD_INDEX))
    assert a.query(L.LBPF_Q_SITES) == b.query(L.LBPF_Q_SITES) == 40 * 37 * 67


def test_vector_step_of_several_domains_and_segments(L, monkeypatch):
    """Two domains in one context, and every item split: same bits as one launch."""
    def make():
        doms = [L.make_domain(nx, ny, nz, lam=10.0, delta=0.4, crystals=[L.make_crystal(**FORM)],
                              **{k: v for k, v in W.C3D_PARAMS.items() if k != "lam"})
                for nx, ny, nz in ((72, 30, 11), (16, 12, 40))]
        s = L.Solver(doms, L.LBPF_D3Q15_D3Q7, L.LBPF_GRAD_DD, L.LBPF_FP32_FP16DEV)
        s.seed([(30.0, 12.0, 5.0, 5.0, 0)], domain=0).seed([(8.0, 6.0, 20.0, 4.0, 0)], domain=1)
        return s
    a, b = both(L, monkeypatch, make)
    a.step(20)
    L.lbpf_set_schedule(a.ctx, 8, 3)
    a.step(20)
    b.step(40)
    for k in (0, 1):
        for x, y in zip(a.fields(k), b.fields(k)):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("shapes,heat_launches", [
    ([(24, 24, 40)] * 5, 1),  # alike: one heat launch
    ([(8, 9, 16), (8, 9, 16), (20, 26, 200), (5, 9, 12), (5, 9, 12)], 3),  # ragged: 2 + 2 + 1
    ([(10, 20, 72, 7), (11, 20, 72, 7), (11, 19, 70, 0)], 2),  # walls and periodic apart
])
def test_heat_launch_over_several_domains(L, monkeypatch, shapes, heat_launches):
    def make():
        doms = [L.make_domain(s[2], s[1], s[0], lam=10.0, delta=0.4, crystals=[L.make_crystal(**FORM)],
                              bc=s[3] if len(s) > 3 else 0, **{k: v for k, v in W.C3D_PARAMS.items() if k != "lam"})
                for s in shapes]
        s = L.Solver(doms, L.LBPF_D3Q15_D3Q7, L.LBPF_GRAD_DD, L.LBPF_FP32_FP16DEV)
        for k, sh in enumerate(shapes):
            s.write_fields(*smooth_fields(sh[:3], k), domain=k)
        return s
    a, b = both(L, monkeypatch, make)
    for n in (1, 4):
        n0 = a.query(L.LBPF_Q_STEP_KERNELS)
        a.step(n)
        b.step(n)
        assert a.query(L.LBPF_Q_STEP_KERNELS) - n0 == n * (heat_launches + 1)
        for k in range(len(shapes)):
            for x, y in zip(a.fields(k), b.fields(k)):
                assert np.array_equal(x, y)


def test_one_launch_step_where_the_work_field_does_not_fit(L, monkeypatch):
    """A state that fits the device memory only without the vector step's work
    field is still taken, and gives the same results."""
    import torch
    n, prm = 256, dict(W.C3D_PARAMS, delta=0.4)
    seeds = [(128.0, 128.0, 128.0, 8.0, 0)]

    def make():
        return gpu_run(L, 1, (n, n, n), prm, [FORM], seeds=seeds, precision=2)
    a, b = both(L, monkeypatch, make)  # both kernels loaded
    a.step(3)
    b.step(3)
    ref = a.fields()
    need = b.query(L.LBPF_Q_DEVICE_BYTES)
    assert a.query(L.LBPF_Q_DEVICE_BYTES) - need > 50e6  # the work field, less a smaller table of items
    a.close()
    b.close()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    hog = torch.empty(int(free - need - 40e6), dtype=torch.uint8, device="cuda")
    monkeypatch.delenv("LBPF_KERNEL")
    s = make()
    del hog
    torch.cuda.empty_cache()
    n0 = s.query(L.LBPF_Q_STEP_KERNELS)
    s.step(3)
    assert s.query(L.LBPF_Q_STEP_KERNELS) - n0 == 3
    for x, y in zip(ref, s.fields()):
        assert np.array_equal(x, y)
