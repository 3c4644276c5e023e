"""Velocities or spins written without positions (no sort follows) reach the pair forces of
the next substep in every form: the run ends with the bits of one that was given them with
the particles.  Contacts with friction make both count."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("what", ["u", "w", "uw"])
def test_written_velocities_reach_the_pairs(form, what):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    n, per = (14, 13, 12), (1, 1, 1)
    rng = np.random.default_rng(8)
    g = np.stack(np.meshgrid(*[np.arange(8)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = 0.5 + 0.97 * g + 0.01 * rng.uniform(-1, 1, g.shape)  # overlapping neighbours
    old = {k: 0.01 * rng.standard_normal(x.shape) for k in "uw"}
    new = {k: 0.01 * rng.standard_normal(x.shape) if k in what else old[k] for k in "uw"}
    out = []
    for late in (False, True):
        dom = dps.Domain(n, per, 0.7, form, max_particles=len(x))
        dom.add_particles(x, 1.0, 2.5, **(old if late else new))
        dom.set_closure(g=(0, 0, 0), fb_mode=0, e_n=0.9, mu_c=0.25, T_c=4.0, h_c=0.3, n_int=1, n_dem=4, skin=0.8,
                        eps_min=0.05, drag=0, pressure=0, added_mass=0)
        dom.prepare()
        if late:
            dom.write_particles(**{k: new[k] for k in what})
        dom.step(1)
        out.append(dom.read_particles())
        dom.close()
    for k in ("x", "u", "w"):
        assert np.array_equal(out[0][k], out[1][k]), k
