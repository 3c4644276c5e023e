"""A launch shape set between two steps leaves the results alone: the lists built under
the shape before it are used under the next one, so tile sizes on and off multiples of
32 follow one another, and every run ends with the bits of the run that kept its shape."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [[], [32, 48], [256, 100, 256], [33, 1000, 64], [128, 40, 32]]


@pytest.mark.parametrize("form", ["f64", "f32", "f16s"])
def test_shape_changes_between_steps(form):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    n, per = (14, 13, 12), (1, 0, 1)
    rng = np.random.default_rng(2)
    g = np.stack(np.meshgrid(np.arange(8), np.arange(7), np.arange(7), indexing="ij"), -1).reshape(-1, 3)
    x = 0.9 + 1.7 * g + 0.2 * rng.uniform(-1, 1, g.shape)
    d, u = rng.uniform(0.9, 1.1, len(x)), 0.01 * rng.standard_normal(x.shape)
    out = []
    for sizes in SIZES:
        b = dps.Batch(form)
        k = b.add_box(n, per, 0.7, max_particles=len(x))
        b.add_particles(k, x, d, np.full(len(x), 2.5), u=u)
        b.set_closure(k, g=(0, 0, -1e-4), e_n=0.9, mu_c=0.25, T_c=4.0, h_c=0.6, h_min=1e-5, n_int=1, n_dem=5, skin=0.7)
        for t in range(4):
            if t and t <= len(sizes):
                b.set_tuning([128, 512, 64, sizes[t - 1], 0])
            b.step(1)
        out.append(b.read_particles(k))
        b.close()
    for r in out[1:]:
        for f in ("x", "u", "w"):
            assert np.array_equal(out[0][f], r[f]), f
