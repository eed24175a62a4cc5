"""Fields of a context with padded rows (the vector step, rows not a multiple of
four sites) between its arrays and the caller's dense ones: pageable and pinned
host memory, device memory at any alignment.  Written and read back as they
are, and without a price beside a context whose rows are dense."""
import time

import numpy as np
import pytest

from test_gpu_forms import L, make  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 2, 9), (3, 5, 63), (5, 7, 65), (40, 37, 67), (17, 301, 130)])
def test_fields_come_back_as_written(L, monkeypatch, shape):  # noqa: F811
    import torch
    monkeypatch.setenv("LBPF_KERNEL", "vector")
    s = make(L, [shape], 2)
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    for where in ("pageable", "pinned", "device", "device + 1 byte"):
        phi, u = (rng.standard_normal(shape).astype(np.float32) for _ in range(2))
        if where == "pageable":
            s.write_fields(phi, u)
            out = np.full(shape, np.nan, np.float32)
            L.lbpf_read_fields(s.ctx, 0, L.LBPF_READ_PHI, out)
        else:
            off = where == "device + 1 byte"

            def tensor(a):
                b = torch.from_numpy(a.view(np.uint8).ravel())
                if where == "pinned":
                    return b.pin_memory()
                t = torch.empty(b.numel() + off, dtype=torch.uint8, device="cuda")
                t[off:] = b.cuda()
                return t[off:]
            L.lbpf_write_fields(s.ctx, 0, tensor(phi), tensor(u))
            t = tensor(np.full(shape, np.nan, np.float32))
            L.lbpf_read_fields(s.ctx, 0, L.LBPF_READ_PHI, t)
            out = t.cpu().numpy().view(np.float32).reshape(shape)
        assert np.array_equal(out, phi), where
        got = s.fields()
        assert np.array_equal(got[0], phi), where
        # u comes back as the sum of its lagged form's parts: one rounding each way
        assert np.all(np.abs(got[1] - u) <= 2.0 ** -23 * (np.abs(u) + np.abs(phi))), where


def test_host_copies_take_no_longer_than_dense_ones(L, monkeypatch):  # noqa: F811
    """207 x 174 x 190 from pinned memory: a pitched copy took 4.8 times the dense one."""
    import torch
    shape = (190, 174, 207)
    phi = torch.zeros(shape).pin_memory()
    best = []
    for kernel in ("vector", "generic"):
        monkeypatch.setenv("LBPF_KERNEL", kernel)
        s = make(L, [shape], 2)
        times = []
        for _ in range(8):
            torch.cuda.synchronize()
            t = time.perf_counter()
            L.lbpf_write_fields(s.ctx, 0, phi, phi)
            times.append(time.perf_counter() - t)
        best.append(min(times))
        s.close()
    assert best[0] <= 2.5 * best[1]
