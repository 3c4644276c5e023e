"""The DEM of boxes with few particles: all substeps of a one-tile box in one launch,
and one launch per substep for tiles of 32 particles with 8 lanes each, against the
general kernels, which the same box takes as part of a larger batch.  Lists, lanes and
orders of a box do not depend on the batch, so the particles end with the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def cluster(n, per, count, seed):
    rng = np.random.default_rng(seed)
    m = int(np.ceil(count ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:count]
    x = 0.45 + g * 1.02 + 0.04 * rng.uniform(-1, 1, (count, 3))  # the first layer near the walls
    u = 0.01 * rng.standard_normal((count, 3))
    u[0] = (0.25, 0.2, 0.22)  # leaves the list's inner shell within a subcycle
    return dict(x=x, d=rng.uniform(0.85, 1.0, count), u=u, w=0.02 * rng.standard_normal((count, 3)))


@pytest.mark.parametrize("form", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("per", [(1, 1, 1), (0, 1, 0)])
@pytest.mark.parametrize("count", [1, 2, 31, 32, 33, 300])
def test_alone_and_in_a_batch(form, per, count):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    n = (14, 13, 12)
    p = cluster(n, per, count, 5 + count)
    kw = dict(g=(0.0, 0.0, -1e-4), fb_mode=0, fb=(0, 0, 0), e_n=0.9, mu_c=0.25, T_c=4.0, h_c=0.5, h_min=1e-5, C_am=0.5,
              n_int=2, n_dem=7, lub_limiter=1, lub_cap=0.25, eps_min=0.05, skin=0.9, drag=0, pressure=0, added_mass=0)
    rng = np.random.default_rng(1)
    other = (30, 30, 30)
    m = 24 ** 3
    g = np.stack(np.meshgrid(*[np.arange(24)] * 3, indexing="ij"), -1).reshape(-1, 3)
    out = []
    for extra in (0, 1):
        b = dps.Batch(form)
        k = b.add_box(n, per, 0.7, max_particles=count)
        b.add_particles(k, p["x"], p["d"], np.full(count, 2.5), u=p["u"], w=p["w"])
        b.set_closure(k, **kw)
        if extra:
            q = b.add_box(other, (1, 1, 1), 0.7, max_particles=m)
            b.add_particles(q, (g + 0.5) * 1.25, np.full(m, 0.8), np.full(m, 2.5),
                            u=0.001 * rng.standard_normal((m, 3)))
            b.set_closure(q, **kw)
        b.step(2)
        out.append(b.read_particles(k))
        b.close()
    for f in ("x", "u", "w"):
        assert np.isfinite(out[0][f]).all()
        assert np.array_equal(out[0][f], out[1][f]), f
