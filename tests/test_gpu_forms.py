"""Which form of the step a context takes (LBPF_Q_STEP_FORM): the bit-for-bit
comparisons of test_gpu_vec.py and test_gpu_tile.py are worth something only
where the two contexts take different forms, and the rules that choose a form
are stated in sizes."""
import pytest

import test_gpu_vec as V
from helpers import gpu_run
from paper_1606_09432_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MARCH, STAGED, VECTOR, TILE = range(4)


@pytest.fixture(scope="module")
def L():
    from paper_1606_09432_gb300 import build as B
    from paper_1606_09432_gb300 import lbpf
    B.build()
    lbpf.load()
    return lbpf


def make(L, shapes, precision, lattice=None, bcs=None):
    """A context of the given (nz, ny, nx) domains, unseeded."""
    d3 = shapes[0][0] > 1
    prm = {k: v for k, v in (W.C3D_PARAMS if d3 else W.C1_PARAMS).items() if k != "lam"}
    cr = L.make_crystal(**(V.FORM if d3 else dict(kind=0, eps=0.05)))
    doms = [L.make_domain(s[2], s[1], s[0], lam=10.0, crystals=[cr], bc=bcs[k] if bcs else 0, **dict(prm, delta=0.4))
            for k, s in enumerate(shapes)]
    return L.Solver(doms, (1 if d3 else 0) if lattice is None else lattice, L.LBPF_GRAD_DD, precision)


def form(L, *args, **kw):
    s = make(L, *args, **kw)
    try:
        return int(s.query(L.LBPF_Q_STEP_FORM))
    finally:
        s.close()


@pytest.mark.parametrize("lattice", [1, 2, 3])
@pytest.mark.parametrize("shape", V.SHAPES + [(9, 14, 74), (40, 37, 67), (256, 256, 256)])
def test_comparisons_of_the_vector_step_compare_two_forms(L, monkeypatch, shape, lattice):
    forms = []
    for kernel in ("vector", "generic"):
        monkeypatch.setenv("LBPF_KERNEL", kernel)
        s = make(L, [shape], 2, lattice)
        n0 = s.query(L.LBPF_Q_STEP_KERNELS)
        s.step(3)
        forms.append((int(s.query(L.LBPF_Q_STEP_FORM)), int(s.query(L.LBPF_Q_STEP_KERNELS) - n0)))
        s.close()
    assert forms == [(VECTOR, 6), (MARCH, 3)]


@pytest.mark.parametrize("precision", range(5))
@pytest.mark.parametrize("shape", [(1, 2, 2), (1, 7, 31), (1, 25, 61), (1, 40, 95), (1, 64, 128)])
def test_comparisons_of_the_one_tile_step_compare_two_forms(L, monkeypatch, shape, precision):
    forms = []
    for kernel in ("", "generic"):
        monkeypatch.setenv("LBPF_KERNEL", kernel)
        forms.append(form(L, [shape], precision))
    assert forms == [TILE, MARCH]


def test_schedule_given_returns_to_the_march(L, monkeypatch):
    monkeypatch.setenv("LBPF_KERNEL", "")
    s = make(L, [(1, 33, 70)], 1)
    assert s.query(L.LBPF_Q_STEP_FORM) == TILE
    L.lbpf_set_schedule(s.ctx, 16, 5)
    assert s.query(L.LBPF_Q_STEP_FORM) == MARCH and s.query(L.LBPF_Q_TILE_ROWS) == 16


def test_cached_2d_schedule_is_taken_again(L, tmp_path, monkeypatch):
    """A schedule timed on the 2D march is cached and read by the next context."""
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("LBPF_TUNE_CACHE", str(cache))
    monkeypatch.setenv("LBPF_KERNEL", "generic")
    monkeypatch.setenv("LBPF_AUTOTUNE", "1")
    s = gpu_run(L, 0, (1, 90, 130), W.C1_PARAMS, [dict(kind=0, eps=0.05)], seeds=[(65.0, 45.0, 0.0, 6.0, 0)], precision=1)
    s.step(2)
    key, v, seg = cache.read_text().split()
    cache.write_text(f"{key} 1 {int(seg) + 3}\n")  # unlike any rule's choice
    monkeypatch.setenv("LBPF_AUTOTUNE", "0")
    s = gpu_run(L, 0, (1, 90, 130), W.C1_PARAMS, [dict(kind=0, eps=0.05)], seeds=[(65.0, 45.0, 0.0, 6.0, 0)], precision=1)
    assert s.query(L.LBPF_Q_TILE_ROWS) == 16 and s.query(L.LBPF_Q_SEGMENT) == int(seg) + 3
    assert s.query(L.LBPF_Q_STEP_FORM) == MARCH


@pytest.mark.parametrize("shapes,bcs,want", [
    ([(64, 64, 64)] * 64, [7 * (k % 2) for k in range(64)], MARCH),  # a heat launch a domain: more than they earn
    ([(64, 64, 64)] * 64, None, VECTOR),
    ([(64, 64, 64)] * 64, [7 * (k // 32) for k in range(64)], VECTOR),
    ([(64, 64, 64), (8, 12, 64)] * 32, None, VECTOR),  # pairs of unlike domains share a launch
    ([(128, 128, 128)] * 8, [7 * (k % 2) for k in range(8)], VECTOR),
])
def test_heat_launches_count_in_the_choice_of_the_vector_step(L, monkeypatch, shapes, bcs, want):
    monkeypatch.setenv("LBPF_KERNEL", "")
    assert form(L, shapes, 2, bcs=bcs) == want


@pytest.mark.parametrize("shape,want", [((500, 2, 512), MARCH), ((1000, 2, 128), MARCH), ((300, 5, 200), MARCH),
                                        ((500, 6, 512), VECTOR), ((256, 13, 256), VECTOR), ((64, 64, 64), VECTOR),
                                        ((400, 400, 40), VECTOR), ((400, 400, 24), MARCH), ((40, 40, 40), MARCH)])
@pytest.mark.parametrize("lattice", [1, 3])
def test_vector_step_where_its_tiles_are_full(L, monkeypatch, shape, lattice, want):
    monkeypatch.setenv("LBPF_KERNEL", "")
    assert form(L, [shape], 2, lattice) == want


BATCHES = [((1, 7, 128), 3000, (MARCH, MARCH, MARCH)), ((1, 128, 128), 200, (None, MARCH, MARCH)),
           ((1, 64, 64), 500, (MARCH, None, MARCH)), ((1, 32, 32), 1000, (MARCH, TILE, TILE)),
           ((1, 256, 256), 30, (TILE, TILE, TILE)), ((1, 64, 64), 1, (TILE, TILE, TILE)), ((1, 2, 2), 1, (TILE, TILE, TILE)),
           ((1, 800, 800), 1, (TILE, TILE, TILE)), ((1, 2048, 2048), 1, (MARCH, TILE, TILE)),
           ((1, 3000, 3000), 1, (MARCH, MARCH, MARCH)), ((1, 100000, 31), 1, (None, TILE, TILE))]


@pytest.mark.parametrize("shape,count,want", BATCHES)
def test_one_tile_step_where_its_tiles_cost_less(L, monkeypatch, shape, count, want):
    """FP64, FP32, FP16; None: over the FP64 limit of sites, or too close to call."""
    monkeypatch.setenv("LBPF_KERNEL", "")
    for precision, w in enumerate(want):
        if w is not None:
            assert form(L, [shape] * count, precision) == w, precision


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_one_tile_step_with_walls(L, monkeypatch, precision):
    monkeypatch.setenv("LBPF_KERNEL", "")
    assert form(L, [(1, 1000, 1000)], precision, bcs=[3]) == TILE
    assert form(L, [(1, 7, 128)] * 1500, precision, bcs=[3] * 1500) == MARCH
