"""Read-back of particles and fields over the sizes of its routes: one copy, the
driver's copy of a single array, and the ring of pinned chunks, which goes round
once 8 MB are in flight.  The device values are known, so the bytes are equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# 12 doubles a particle: one copy (< 2 MB), chunks that all fit, the ring
@pytest.mark.parametrize("count", [1, 500, 21845, 21846, 80000, 87382, 300001])
def test_particles_come_back_as_written(count):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    n = (48, 45, 51)
    rng = np.random.default_rng(count)
    x, u, w = rng.random((count, 3)) * n, rng.standard_normal((count, 3)), rng.standard_normal((count, 3))
    dom = dps.Domain(n, (1, 1, 1), 0.7, "f64", max_particles=count)
    dom.add_particles(x, 0.5, 2.5, u=u, w=w)
    for _ in range(2):
        got = dom.read_particles()
        for k, v in (("x", x), ("u", u), ("w", w)):
            assert np.array_equal(got[k], v), k
    dom.close()


# f_pf alone: the driver's copy (up to 24 MB) and the ring
@pytest.mark.parametrize("n", [(3, 4, 5), (64, 33, 16), (104, 100, 101), (128, 120, 100)])
def test_fields_come_back_as_written(n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    rng = np.random.default_rng(1)
    dom = dps.Domain(n, (1, 1, 1), 0.7, "f64")
    shape = dom.read_fields(("f_pf",))["f_pf"].shape
    f = rng.standard_normal(shape)
    dom.write_fields(f_pf=f)
    for names in (("f_pf",), ("f_pf", "eps_f")):
        assert np.array_equal(dom.read_fields(names)["f_pf"], f)
    dom.close()
