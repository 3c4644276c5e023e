"""The bricks of the step's fluid fields over axes of more than 2^21 cells: grad P and the
convective Du_f/Dt of every cell against plain sums (tolerances of the same comparison for
small boxes: 1e-15 and 6e-7 of the density, 2e-14 and 5e-6 of the velocity)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,tp,tu", [("f64", 1e-15, 2e-14), ("f32", 6e-7, 5e-6)])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_fields_beyond_two_million_cells(axis, form, tp, tu):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    n = [1, 1, 1]
    n[axis] = nc = (1 << 21) + 39
    c, w = dps.lattice()
    rng = np.random.default_rng(5)
    u = 0.01 * rng.uniform(-1, 1, (3, nc))
    f = np.empty((19, nc))
    rho = rng.uniform(0.9, 1.1, nc)
    for q in range(19):
        f[q] = w[q] * rho * (1 + 3 * (c[q] @ u))
    dom = dps.Domain(n, (1, 1, 1), 0.7, form)
    dom.set_closure(g=(0, 0, 0), fb_mode=0, n_int=1, n_dem=1)
    dom.write_pdfs(f)
    f = dom.read_pdfs()
    dom.step(1)
    got = dom.read_fields(("gradP", "DuDt"))
    dom.close()
    rho = f.sum(0)
    u = (c.T @ f) / rho
    # the other axes are one cell: sum_q w_q c_q phi(x + c_q) = (phi(x+1) - phi(x-1)) / 6 along this one
    d = lambda p: (np.roll(p, -1) - np.roll(p, 1)) / 6
    gp = np.zeros((3, nc))
    gp[axis] = d(rho)
    assert np.abs(got["gradP"] - gp).max() <= tp * rho.max()
    conv = np.array([3 * u[axis] * d(u[b]) for b in range(3)])
    assert np.abs(got["DuDt"] - conv).max() <= tu * np.abs(u).max()
