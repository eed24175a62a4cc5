"""The heat catch-up of contexts whose domains differ widely in size: the large
domain's share of the launch does not shrink with the number of small ones."""
import time

import numpy as np
import pytest

from test_gpu_forms import L, make  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_catch_up_time_does_not_depend_on_the_number_of_small_domains(L):  # noqa: F811
    """256^3 FP32 beside three or four domains of 16^3: four took 2.1 times as long."""
    import torch
    out = torch.empty((16, 16, 16), device="cuda")
    best = []
    for small in (3, 4):
        s = make(L, [(256, 256, 256)] + [(16, 16, 16)] * small, 1)
        times = []
        for _ in range(8):
            s.step(1)
            torch.cuda.synchronize()
            t = time.perf_counter()
            L.lbpf_read_field(s.ctx, 1, L.LBPF_FIELD_U, out)
            times.append(time.perf_counter() - t)
        best.append(min(times))
        s.close()
    assert best[1] <= 1.5 * best[0]


@pytest.mark.parametrize("precision", [0, 1])
def test_catch_up_of_unlike_domains(L, precision):  # noqa: F811
    """Seven domains, one large: each reads as it does alone."""
    shapes = [(5, 6, 7)] * 3 + [(40, 90, 110)] + [(2, 3, 4)] * 3
    dtype = np.float64 if precision == 0 else np.float32
    rng = np.random.default_rng(precision)
    fields = [(np.tanh(rng.standard_normal(s)).astype(dtype), (0.1 * rng.standard_normal(s)).astype(dtype)) for s in shapes]
    a = make(L, shapes, precision)
    for k, f in enumerate(fields):
        a.write_fields(*f, domain=k)
    a.step(3)
    for k, f in enumerate(fields):
        b = make(L, [shapes[k]], precision)
        b.write_fields(*f)
        b.step(3)
        for x, y in zip(a.fields(k), b.fields()):
            assert np.array_equal(x, y)
        b.close()
