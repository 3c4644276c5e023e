"""FP64 fluid kernels where their fixed-point and FP64 paths meet: the relaxation
against the CPU oracle with populations, porosities and forces inside, across and
outside the fixed-point ranges (mixed in one box, both parities, walls), and the
step's grad P and Du_f/Dt against plain FP64 sums, for velocities of any size.

Tolerances.  Relaxation: the oracle rounds ~6 operations of values up to the
largest population, 1e-15 of it bounds them twice over; the next steps add as
much each.  grad P sums 18 terms of weight at most 1/18: 18 x 2^-53 / 18 x 8 < 1e-15
of the largest density.  Du_f/Dt: u carries 19 roundings (2e-15), its gradient
as many, so 3 u . grad u is good to ~5 x 2e-15 of u_max x (u_max + 1): 2e-14 u_max.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _populations(c, w, nc, scale, speed, noise, seed):
    rng = np.random.default_rng(seed)
    u = speed * rng.uniform(-1, 1, (3, nc))
    cu = c @ u
    rho = scale * rng.uniform(0.9, 1.1, nc)
    return w[:, None] * rho * (1 + 3 * cu + 4.5 * cu ** 2 - 1.5 * (u ** 2).sum(0)) * (1 + noise * rng.standard_normal((19, nc)))


RANGES = {  # density, velocity, noise, porosity range, f_pf
    "inside": (1.0, 0.05, 1e-3, (0.3, 1.0), 1e-4),
    "low_density": (0.5, 0.02, 1e-3, (0.3, 1.0), 1e-4),   # across rho = 1/2
    "high_density": (1.7, 0.05, 1e-2, (0.3, 1.0), 1e-4),  # populations across 1/2, 1/8, 1/16
    "fast": (1.0, 0.2, 1e-3, (0.3, 1.0), 1e-4),           # across |j| = 1/8
    "dense_solid": (1.0, 0.05, 1e-3, (0.1, 0.15), 1e-4),  # across eps = 1/8
    "strong_force": (1.0, 0.05, 1e-3, (0.3, 1.0), 0.1),   # across |f_pf| = 1/8
    "far_outside": (3.0, 0.3, 1e-1, (0.05, 1.0), 0.5),
}


@pytest.mark.parametrize("tau", [0.5045, 0.9, 3.0])
@pytest.mark.parametrize("name", list(RANGES))
def test_relaxation_across_the_fixed_point_ranges(name, tau):
    _need_gpu()
    import oracle as O
    from paper_1711_00336_gb300 import dps
    scale, speed, noise, er, fa = RANGES[name]
    n, per = (13, 6, 9), (1, 0, 1)
    nc = n[0] * n[1] * n[2]
    c, w = dps.lattice()
    co, _, _ = O.lattice()
    perm = [next(k for k in range(19) if (co[k] == c[q]).all()) for q in range(19)]  # library plane -> oracle plane
    rng = np.random.default_rng(len(name))
    f = _populations(c, w, nc, scale, speed, noise, seed=len(name))
    eps, fpf = rng.uniform(*er, nc), fa * rng.standard_normal((3, nc))
    dom = dps.Domain(n, per, tau, "f64")
    dom.write_pdfs(f)
    dom.write_fields(eps_f=eps, f_pf=fpf)
    P = O.make_params(n, per, tau)
    ref = np.empty_like(f)
    ref[perm] = f
    for step in (1, 2):
        try:
            dom.collide_stream(1)
        except dps.DPSError:
            assert name in ("far_outside", "strong_force")  # a density below zero: the run stops
            break
        ref = O.collide_stream(P, ref, eps, fpf)
        got = dom.read_pdfs()
        assert np.abs(got - ref[perm]).max() <= step * 1e-15 * max(1.0, np.abs(ref).max() / eps.min()), step
    dom.close()


@pytest.mark.parametrize("vk", [dict(eilers=1), dict(smagorinsky=1), dict(eilers=1, smagorinsky=1)],
                         ids=["eilers", "smagorinsky", "both"])
@pytest.mark.parametrize("name", list(RANGES))
def test_cell_viscosity_across_the_fixed_point_ranges(name, vk):
    """The same with a relaxation time per cell.  omega's own rounding (twenty
    operations) multiplies f - f_eq, below the largest population: 5e-15."""
    _need_gpu()
    import oracle as O
    from paper_1711_00336_gb300 import dps
    scale, speed, noise, er, fa = RANGES[name]
    n, per, tau = (13, 6, 9), (1, 0, 1), 0.55
    nc = n[0] * n[1] * n[2]
    c, w = dps.lattice()
    co, _, _ = O.lattice()
    perm = [next(k for k in range(19) if (co[k] == c[q]).all()) for q in range(19)]
    rng = np.random.default_rng(len(name))
    f = _populations(c, w, nc, scale, speed, noise, seed=len(name))
    eps, fpf = rng.uniform(*er, nc), fa * rng.standard_normal((3, nc))
    dom = dps.Domain(n, per, tau, "f64")
    dom.set_closure(g=(0, 0, 0), fb_mode=0, fb=(0, 0, 0), n_int=1, n_dem=1, **vk)
    dom.prepare()
    dom.write_pdfs(f)
    dom.write_fields(eps_f=eps, f_pf=fpf)
    P = O.make_params(n, per, tau, n_int=1, n_dem=1, **vk)
    ref = np.empty_like(f)
    ref[perm] = f
    for step in (1, 2):
        try:
            dom.collide_stream(1)
        except dps.DPSError:
            assert name in ("far_outside", "strong_force")
            break
        ref = O.collide_stream(P, ref, eps, fpf)
        got = dom.read_pdfs()
        assert np.abs(got - ref[perm]).max() <= step * 5e-15 * max(1.0, np.abs(ref).max() / eps.min()), step
    dom.close()


def test_non_finite_populations_are_reported():
    _need_gpu()
    from paper_1711_00336_gb300 import dps
    c, w = dps.lattice()
    f = np.tile(w[:, None], (1, 5 * 4 * 3))
    f[3, 17] = np.nan
    dom = dps.Domain((5, 4, 3), (1, 1, 1), 0.7, "f64")
    dom.write_pdfs(f)
    with pytest.raises(dps.DPSError, match="UNSTABLE"):
        dom.collide_stream(1)
    dom.close()


@pytest.mark.parametrize("speed", [1e-6, 1e-2, 0.2])
@pytest.mark.parametrize("n,per", [((8, 8, 8), (1, 1, 1)), ((17, 9, 3), (1, 0, 1)), ((1, 2, 40), (1, 1, 0))])
def test_step_gradients_against_plain_sums(n, per, speed):
    _need_gpu()
    from paper_1711_00336_gb300 import dps
    nc = n[0] * n[1] * n[2]
    c, w = dps.lattice()
    f = _populations(c, w, nc, 1.0, speed, 0.1 * speed, seed=5)
    dom = dps.Domain(n, per, 0.7, "f64")
    dom.set_closure(g=(0, 0, 0), fb_mode=0, fb=(0, 0, 0), n_int=1, n_dem=1)
    dom.write_pdfs(f)
    dom.step(1)
    got = dom.read_fields(("gradP", "DuDt"))
    dom.close()
    rho = f.sum(0)
    u = (c.T @ f) / rho
    idx = np.arange(nc).reshape(n[2], n[1], n[0])

    def nb(q):
        i = idx
        for a in range(3):
            k = np.arange(n[a]) + c[q][a]
            k = k % n[a] if per[a] else np.clip(k, 0, n[a] - 1)
            i = np.take(i, k, axis=2 - a)
        return i.ravel()

    def grad(p):
        return sum(w[q] * 3 * np.outer(c[q], p[nb(q)]) for q in range(1, 19))

    gp = grad(rho) / 3
    conv = np.array([(u * grad(u[b])).sum(0) for b in range(3)])
    assert np.abs(got["gradP"] - gp).max() <= 1e-15 * rho.max()
    assert np.abs(got["DuDt"] - conv).max() <= 2e-14 * np.abs(u).max()


@pytest.mark.parametrize("form", ["f32", "f16s"])
@pytest.mark.parametrize("steps", [0, 1])
@pytest.mark.parametrize("n,per", [((8, 8, 8), (1, 1, 1)), ((17, 9, 4), (1, 1, 1)), ((6, 5, 7), (1, 0, 0)),
                                   ((5, 3, 7), (0, 1, 1)), ((2, 9, 3), (0, 1, 1))])
def test_fp32_moments_and_gradients(form, steps, n, per):
    """The cell pairs of the moments pass (even and odd nx and cell counts, both
    parities, walls) and the staged gradients.  rho carries 19 roundings of a sum
    below 0.3 and that of 1 + s: 4e-7; grad P adds 18 terms, sum |w c| = 1/3: 6e-7."""
    _need_gpu()
    from paper_1711_00336_gb300 import dps
    nc = n[0] * n[1] * n[2]
    c, w = dps.lattice()
    dom = dps.Domain(n, per, 0.7, form)
    dom.set_closure(g=(0, 0, 0), fb_mode=0, fb=(0, 0, 0), n_int=1, n_dem=1)
    dom.write_pdfs(_populations(c, w, nc, 1.0, 1e-2, 1e-2, seed=7))
    if steps:
        dom.step(steps)
    f = dom.read_pdfs()
    dom.step(1)
    got = dom.read_fields(("gradP", "DuDt"))
    dom.close()
    rho = f.sum(0)
    idx = np.arange(nc).reshape(n[2], n[1], n[0])

    def nb(q):
        i = idx
        for a in range(3):
            k = np.arange(n[a]) + c[q][a]
            k = k % n[a] if per[a] else np.clip(k, 0, n[a] - 1)
            i = np.take(i, k, axis=2 - a)
        return i.ravel()

    gp = sum(w[q] * np.outer(c[q], rho[nb(q)]) for q in range(1, 19))
    assert np.abs(got["gradP"] - gp).max() <= 6e-7 * rho.max()
    if not steps:  # no u_prev yet: the convective term alone; u good to 4e-7, its gradient to 1e-6
        u = (c.T @ f) / rho
        conv = np.array([(u * sum(3 * w[q] * np.outer(c[q], u[b][nb(q)]) for q in range(1, 19))).sum(0)
                         for b in range(3)])
        assert np.abs(got["DuDt"] - conv).max() <= 5e-6 * np.abs(u).max()
