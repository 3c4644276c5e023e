"""Lubrication with a wall in the FP64 form without the limiter, for small and large spheres
and gaps down to 1e-5 in boxes on both sides of 512 cells: one substep against the formula.

The gap x - d/2 is one exact subtraction, so the change of the velocity, u b dt/m, carries
the roundings of the coefficient b, the mass and the update only: less than 15 of 2^-53 on
either side, 4e-15 together."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("gap", [1e-5, 1e-3, 1e-2])
@pytest.mark.parametrize("d0", [0.3, 0.9, 1.4])
@pytest.mark.parametrize("nz", [64, 600])
def test_wall_lubrication_near_contact(nz, d0, gap, side):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    n, tau, rho_p = (24, 24, nz), 0.55, 2.5
    rng = np.random.default_rng(4)
    xy = 2.0 + 4.0 * np.stack(np.meshgrid(np.arange(6), np.arange(6), indexing="ij"), -1).reshape(-1, 2)
    k = len(xy)
    d, h = d0 * rng.uniform(0.95, 1.0, k), gap * rng.uniform(1.0, 2.0, k)
    z = nz - (0.5 * d + h) if side else 0.5 * d + h
    u = 1e-7 * rng.uniform(0.5, 1.5, (k, 3))
    dom = dps.Domain(n, (1, 1, 0), tau, "f64", max_particles=k)
    dom.add_particles(np.column_stack([xy, z]), d, rho_p, u=u)
    dom.set_closure(g=(0, 0, 0), fb_mode=0, h_c=0.5, h_min=1e-6, n_int=1, n_dem=1, skin=0.8, lub_limiter=0, drag=0,
                    pressure=0, added_mass=0)
    dom.step(1)
    got = dom.read_particles()["u"] - u
    dom.close()
    h = (nz - z if side else z) - 0.5 * d
    mu, dm, m = (tau - 0.5) / 3, 2 * d, rho_p * np.pi / 6 * d ** 3
    r = dm / h
    L = np.log(r / 2)
    sq = 1.5 * np.pi * mu * dm * (r / 4 + 18 / 40 * L + 9 / 84 * L / r)
    sh = 0.5 * np.pi * mu * dm * L
    ref = -np.column_stack([sh, sh, sq]) / m[:, None] * u
    assert np.abs(got / ref - 1).max() <= 4e-15
