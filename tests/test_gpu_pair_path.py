"""FP64 DEM pair kernel against the CPU oracle where its two ways of evaluating a
pair (64-bit integers for lubrication, the FP64 body for the rest) meet: the
position scales of boxes below and above 512 cells, boxes and diameters outside
the integer path, gaps at the floor, the limiter and the cut-off, tiles with more
overlapping pairs than the block's queue holds, and either law switched off.

Tolerance: an uncapped coefficient varies by d(gap)/gap; the distance of two
spheres carries an FP64 rounding of ~4e-16 and the limiter caps gaps below
~1e-3, so a pair's force is good to ~4e-13 and a step of ten substeps to ~4e-12
of the largest velocity; 1e-10 leaves a factor of 25 for cancelling sums.
"""
import numpy as np
import pytest


pytestmark = pytest.mark.gpu
TOL = 1e-10


def lattice(n, per, spacing, d, jitter, seed, cluster=1):
    rng = np.random.default_rng(seed)
    m = [max(1, int((n[a] - (0 if per[a] else 0.2)) / spacing)) for a in range(3)]
    g = np.stack(np.meshgrid(*[np.arange(k) for k in m], indexing="ij"), -1).reshape(-1, 3)
    x = (g + 0.5) * spacing + (0 if all(per) else 0.1) + jitter * rng.uniform(-1, 1, g.shape)
    if cluster > 1:
        x = np.repeat(x, cluster, 0) + rng.uniform(-0.12, 0.12, (len(x) * cluster, 3))
    x = np.where(per, np.mod(x, n), x)
    k = len(x)
    return dict(x=x, u=0.01 * rng.standard_normal((k, 3)), w=0.01 * rng.standard_normal((k, 3)),
                d=np.broadcast_to(d, k) * rng.uniform(0.97, 1.0, k), rho_p=rng.uniform(2.0, 3.0, k))


CASES = {
    # touching lattice neighbours: gaps around zero, the floor and the limiter
    "near_contact": ((14, 13, 12), (1, 1, 1), dict(spacing=1.0, d=1.0, jitter=0.02), dict(h_c=1.0)),
    "floor_h_min": ((14, 13, 12), (1, 1, 1), dict(spacing=1.0, d=1.0, jitter=0.01), dict(h_c=0.5, h_min=0.02)),
    # the cut-off inside the shell of lattice neighbours, and below any gap
    "cut_off": ((14, 13, 12), (1, 1, 1), dict(spacing=1.3, d=1.0, jitter=0.1), dict(h_c=0.3)),
    "no_cut_off": ((12, 12, 12), (1, 1, 1), dict(spacing=1.0, d=1.0, jitter=0.03), dict(h_c=0.0)),
    # every position scale, and a box past them (FP64 body for all pairs)
    "long_511": ((511, 5, 5), (1, 1, 1), dict(spacing=1.2, d=1.1, jitter=0.06), dict(h_c=0.5)),
    "long_512": ((5, 512, 5), (1, 0, 1), dict(spacing=1.2, d=1.1, jitter=0.06), dict(h_c=0.5)),
    "long_1001": ((5, 5, 1001), (1, 1, 1), dict(spacing=1.25, d=1.1, jitter=0.06), dict(h_c=0.5)),
    # diameters at and below the range of the integer path
    "small_0.26": ((6, 6, 6), (1, 1, 0), dict(spacing=0.3, d=0.268, jitter=0.01), dict(h_c=0.2, eps_min=0.01)),
    "small_0.24": ((6, 6, 6), (1, 1, 0), dict(spacing=0.3, d=0.24, jitter=0.01), dict(h_c=0.2, eps_min=0.01)),
    # clusters of 40 overlapping spheres: more such pairs than a tile's queue holds
    "clusters": ((12, 12, 12), (1, 1, 1), dict(spacing=4.0, d=0.3, jitter=0.0, cluster=40), dict(h_c=0.3, T_c=200.0)),
    "contact_off": ((12, 12, 12), (1, 1, 1), dict(spacing=1.0, d=1.0, jitter=0.03), dict(h_c=0.5, contact=0)),
    "lubrication_off": ((12, 12, 12), (1, 1, 1), dict(spacing=1.0, d=1.0, jitter=0.03), dict(h_c=0.5, lubrication=0)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_fp64_pairs_against_the_oracle(name):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_1711_00336_gb300 import dps
    n, per, lat, more = CASES[name]
    p = lattice(np.array(n, float), np.array(per), seed=len(name), **lat)
    kw = dict(g=(0.0, 0.0, -1e-4), e_n=0.9, mu_c=0.25, T_c=2.0, h_min=1e-5, C_am=0.5, n_int=1, n_dem=10, lub_limiter=1,
              lub_cap=0.25, eps_min=0.05)
    kw.update(more)
    tau = 0.7
    dom = dps.Domain(n, per, tau, "f64", max_particles=len(p["x"]))
    dom.add_particles(p["x"], p["d"], p["rho_p"], u=p["u"], w=p["w"])
    dom.set_closure(fb_mode=0, fb=(0, 0, 0), skin=0.6, drag=0, pressure=0, added_mass=0, **kw)
    dom.step(1)
    got = dom.read_particles()
    st = dom.stats()
    dom.close()
    P = O.make_params(n, per, tau, drag=0, pressure=0, added_mass=0, **kw)
    ref = O.Domain(P, x=p["x"], u=p["u"], w=p["w"], d=p["d"], rho_p=p["rho_p"])
    ref.step(1)
    r = ref.particles()
    for k in ("u", "w"):
        assert np.abs(got[k] - r[k]).max() <= TOL * np.abs(r[k]).max(), k
    dx = got["x"] - r["x"]
    dx -= np.where(per, n, 0) * np.round(dx / np.array(n))
    assert np.abs(dx).max() <= TOL * np.abs(r["u"]).max()
    assert st["status"] == 0


@pytest.mark.parametrize("per", [(0, 1, 1), (1, 0, 0), (0, 0, 0)])
@pytest.mark.parametrize("gap", [-0.1, -1e-6, 1e-7, 9e-6, 1e-4, 0.03, 0.499, 0.501])
def test_fp64_walls_against_the_oracle(per, gap):
    """One sphere at each face (gaps from overlap over the floor, the limiter
    and the cut-off to beyond it), each far from the others."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_1711_00336_gb300 import dps
    n = (14, 15, 13)
    rng = np.random.default_rng(7)
    d = rng.uniform(0.9, 1.6, 6)
    x = np.tile(np.array(n) / 2.0, (6, 1))
    for f in range(6):
        near = gap + 0.5 * d[f]
        x[f, f // 2] = n[f // 2] - near if f % 2 else near
    u, w = 0.01 * rng.standard_normal((6, 3)), 0.01 * rng.standard_normal((6, 3))
    kw = dict(g=(0.0, 0.0, -1e-4), e_n=0.9, mu_c=0.25, T_c=20.0, h_c=0.5, h_min=1e-5, C_am=0.5, n_int=1, n_dem=10,
              lub_limiter=1, lub_cap=0.25, eps_min=0.05)
    dom = dps.Domain(n, per, 0.7, "f64", max_particles=6)
    dom.add_particles(x, d, 2.5, u=u, w=w)
    dom.set_closure(fb_mode=0, fb=(0, 0, 0), skin=0.6, drag=0, pressure=0, added_mass=0, **kw)
    dom.step(1)
    got = dom.read_particles()
    dom.close()
    P = O.make_params(n, per, 0.7, drag=0, pressure=0, added_mass=0, **kw)
    ref = O.Domain(P, x=x, u=u, w=w, d=d, rho_p=np.full(6, 2.5))
    ref.step(1)
    r = ref.particles()
    for k in ("u", "w"):
        assert np.abs(got[k] - r[k]).max() <= TOL * np.abs(r[k]).max(), k


@pytest.mark.parametrize("fast", [0.0, 0.3])
def test_written_velocities_and_moves_beyond_the_inner_shell(fast):
    """Velocities written between sorts reach the pairs, and particles that
    leave the list's inner shell within a subcycle (0.3 cells per step against
    0.05) still meet every partner."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_1711_00336_gb300 import dps
    n, per = (14, 13, 12), (1, 0, 1)
    p = lattice(np.array(n, float), np.array(per), seed=3, spacing=1.35, d=1.0, jitter=0.15)
    u = p["u"].copy()
    u[::17, 0] += fast
    kw = dict(g=(0.0, 0.0, -1e-4), e_n=0.9, mu_c=0.25, T_c=2.0, h_c=0.5, h_min=1e-5, C_am=0.5, n_int=1, n_dem=20,
              lub_limiter=1, lub_cap=0.25, eps_min=0.05)
    dom = dps.Domain(n, per, 0.7, "f64", max_particles=len(p["x"]))
    dom.add_particles(p["x"], p["d"], p["rho_p"], u=p["u"], w=p["w"])
    dom.set_closure(fb_mode=0, fb=(0, 0, 0), skin=0.8, drag=0, pressure=0, added_mass=0, **kw)
    dom.prepare()
    dom.write_particles(u=u)
    dom.step(1)
    got = dom.read_particles()
    dom.close()
    P = O.make_params(n, per, 0.7, drag=0, pressure=0, added_mass=0, **kw)
    ref = O.Domain(P, x=p["x"], u=u, w=p["w"], d=p["d"], rho_p=p["rho_p"])
    ref.step(1)
    r = ref.particles()
    for k in ("u", "w"):
        assert np.abs(got[k] - r[k]).max() <= TOL * np.abs(r[k]).max(), k


@pytest.mark.parametrize("form", ["f64", "f16s"])
@pytest.mark.parametrize("extra", [0, 3000])
def test_outer_pairs_add_nothing_to_slow_particles(form, extra):
    """A lone fast sphere makes every substep after the first visit the outer
    pairs of the list; the other spheres, all slow, end with the same bits (the
    FP32 form deals the entries to its lanes anew, so its sums round anew).
    (extra: enough spheres that a particle is given fewer lanes.)"""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    n, per = (14, 13, 40) if not extra else (26, 25, 40), (1, 1, 1)
    p = lattice(np.array((n[0], n[1], 20 if not extra else 26), float), np.array(per), seed=4, spacing=1.25, d=1.0,
                jitter=0.11)
    assert len(p["x"]) > extra
    kw = dict(g=(0.0, 0.0, -1e-4), fb_mode=0, fb=(0, 0, 0), e_n=0.9, mu_c=0.25, T_c=2.0, h_c=0.5, h_min=1e-5, C_am=0.5,
              n_int=1, n_dem=8, lub_limiter=1, lub_cap=0.25, eps_min=0.05, skin=0.8, drag=0, pressure=0, added_mass=0)
    out = []
    for speed in (0.0, 0.35):
        x = np.vstack([p["x"], [[n[0] / 2, n[1] / 2, 33.0]]])
        u = np.vstack([p["u"], [[speed, 0.0, 0.0]]])
        w = np.vstack([p["w"], [[0.0, 0.0, 0.0]]])
        dom = dps.Domain(n, per, 0.7, form, max_particles=len(x))
        dom.add_particles(x, np.append(p["d"], 1.0), np.append(p["rho_p"], 2.5), u=u, w=w)
        dom.set_closure(**kw)
        dom.step(1)
        out.append(dom.read_particles())
        dom.close()
    for k in ("x", "u", "w"):
        assert np.array_equal(out[0][k][:-1], out[1][k][:-1]), k
