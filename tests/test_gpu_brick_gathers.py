"""The cell gathers (eps_f and the reaction densities) over bricks of 8^3 cells:
boxes smaller than a brick, remainders, one particle, empty bricks, and bricks with
more particles than the stage holds (the walk over global memory), against the CPU
oracle, for the FP64 and the FP32 form.

Tolerance, relative to the largest value: a cell sums at most ~100 products of
three weights and a value, so FP64 rounds by less than 110 x 2^-53 = 1.2e-14 and
FP32 by 110 x 2^-24 = 6.6e-6; the forces behind the reactions add the
interpolations of 27 cells and the drag law (x 10): 1e-12 and 1e-4.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# tau 0.52: the drag of the smallest spheres relaxes by half a step
CASES = {
    "tiny_3_4_5": ((3, 4, 5), (1, 1, 1), 6, (0.3, 0.4)),
    "tiny_walls": ((4, 3, 9), (1, 0, 1), 8, (0.3, 0.4)),
    "one_particle": ((17, 16, 9), (1, 1, 0), 1, (0.8, 0.8)),
    "remainders": ((9, 23, 17), (1, 1, 0), 500, (0.7, 1.1)),
    "fp64_stage_edge": ((16, 16, 16), (1, 1, 1), 1835, (0.5, 0.6)),   # ~448 in 1000 halo cells
    "fp32_stage_edge": ((16, 16, 16), (1, 1, 1), 2884, (0.5, 0.55)),  # ~704
    "over_the_stage": ((16, 8, 24), (1, 1, 1), 6000, (0.3, 0.35)),
    "half_empty": ((32, 16, 16), (1, 1, 1), 900, (0.7, 0.8)),
    # dilute boxes (on average under 120 per brick and halo) with a dense
    # corner: bricks over the small stage, in slabs and over the slabs' size
    "dilute": ((24, 21, 18), (1, 1, 0), 700, (0.7, 1.1)),
    "dilute_slabs": ((48, 47, 46), (1, 1, 1), 1500, (0.5, 0.6)),
    "dilute_walk": ((48, 47, 46), (1, 1, 1), 3500, (0.4, 0.45)),
}


@pytest.mark.parametrize("form,teps,tforce", [("f64", 1.2e-14, 1e-12), ("f32", 6.6e-6, 1e-4)])
@pytest.mark.parametrize("name", list(CASES))
def test_gathers_against_the_oracle(name, form, teps, tforce):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_1711_00336_gb300 import dps
    n, per, count, d = CASES[name]
    rng = np.random.default_rng(len(name))
    L = np.array(n, float)
    if name == "half_empty":
        L[0] /= 2
    if name.startswith("dilute_"):
        L[:] = 16.0
    lo = np.where(per, 0.0, 0.6)
    x = lo + rng.random((count, 3)) * (L - 2 * lo)
    dia = rng.uniform(*d, count)
    u = 0.01 * rng.standard_normal((count, 3))
    kw = dict(g=(0.0, 0.0, -1e-3), e_n=0.9, mu_c=0.25, T_c=1.0, h_c=0.0, h_min=1e-5, C_am=0.5, n_int=1, n_dem=1,
              contact=0, lubrication=0, eps_min=0.02)
    dom = dps.Domain(n, per, 0.52, form, max_particles=count)
    dom.add_particles(x, dia, np.full(count, 2.5), u=u)
    dom.set_closure(fb_mode=0, fb=(0, 0, 0), skin=0.5, **kw)
    dom.prepare()
    eps0 = dom.read_fields(("eps_f",))["eps_f"]
    dom.step(2)  # the second step has an added-mass force
    f = dom.read_fields(("eps_f", "f_pf"))
    dom.close()
    P = O.make_params(n, per, 0.52, **kw)
    ref = O.Domain(P, x=x, u=u, w=np.zeros_like(u), d=dia, rho_p=np.full(count, 2.5))
    e0 = ref.fields()["eps_f"].copy()
    ref.step(2)
    r = dict(eps_f=ref.fields()["eps_f"], f_pf=ref.fpf)
    assert np.abs(eps0 - e0).max() <= teps
    assert np.abs(f["eps_f"] - r["eps_f"]).max() <= tforce
    assert np.abs(f["f_pf"] - r["f_pf"]).max() <= tforce * np.abs(r["f_pf"]).max()
