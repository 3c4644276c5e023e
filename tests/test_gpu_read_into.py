"""dps_read_fields and dps_read_particles into memory of the caller's: pinned, pageable pages
that exist, pages not touched yet, odd offsets, over the sizes of the read-back's routes.  A
large field goes into existing pages by a plain copy, after the staging buffer is mapped and
the field converted (1.6 times the copy alone; by the ring of chunks 3.4 times): 2.5 is allowed."""
import ctypes
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _torch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("kind", ["pinned", "pageable", "fresh", "odd"])
@pytest.mark.parametrize("n", [(3, 4, 5), (64, 64, 64), (128, 120, 100)])
def test_fields_into_the_callers_memory(kind, n):
    torch = _torch()
    from paper_1711_00336_gb300 import dps
    nc = n[0] * n[1] * n[2]
    f = np.random.default_rng(1).standard_normal((3, nc))
    dom = dps.Domain(n, (1, 1, 1), 0.7, "f64")
    dom.write_fields(f_pf=f)
    t = torch.empty(3 * nc + 1, dtype=torch.float64, pin_memory=kind == "pinned")
    if kind in ("pageable", "odd"):
        t.zero_()
    o = int(kind == "odd")
    p = ctypes.cast(t.data_ptr() + 8 * o, ctypes.POINTER(ctypes.c_double))
    dom._ck(dps.lib().dps_read_fields(dom.h, 0x040, p, 3 * nc))
    assert np.array_equal(t.numpy()[o:o + 3 * nc].reshape(3, nc), f)
    dom.close()


@pytest.mark.parametrize("pinned", [True, False])
def test_large_field_into_existing_pages(pinned):
    torch = _torch()
    from paper_1711_00336_gb300 import dps
    n = (192, 192, 192)
    nc = n[0] * n[1] * n[2]
    dom = dps.Domain(n, (1, 1, 1), 0.7, "f64")
    t = torch.zeros(3 * nc, dtype=torch.float64).pin_memory() if pinned else torch.zeros(3 * nc, dtype=torch.float64)
    dev = torch.randn(3 * nc, dtype=torch.float64, device="cuda")
    t.copy_(dev)
    p = ctypes.cast(t.data_ptr(), ctypes.POINTER(ctypes.c_double))

    def best(fn):
        ts = []
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            fn()
            torch.cuda.synchronize()
            ts.append(time.perf_counter() - t0)
        return min(ts)

    plain = best(lambda: t.copy_(dev))
    read = best(lambda: dom._ck(dps.lib().dps_read_fields(dom.h, 0x040, p, 3 * nc)))
    dom.close()
    assert read <= 2.5 * plain, (read, plain)
