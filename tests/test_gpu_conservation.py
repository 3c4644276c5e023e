"""Mass and momentum of an FP64 collide-stream step with exact sums over two million
cells in motion, so that a rounding of one sign would show (over thousands of steps of
a large box it adds up; cells in motion round independently of one another).

Tolerance: a step rounds the 19 populations of a cell, half a unit in the last place
at most and uniform below it; with f_0 in [1/4, 1/2), the axes in [2^-5, 2^-4) and the
diagonals in [2^-6, 2^-5) the changes have variances (2^-54)^2/12, (2^-57)^2/12 and
(2^-58)^2/12: 1.7e-17 for the mass of a cell and 4.1e-18 for a component of its momentum.
The mean over N cells of a step (an even or an odd one) has these over sqrt(N); six times
that is allowed.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def exact_sum(f, w):
    """sum(f - w) in units of 2^-62: every f is a multiple of that and below 1."""
    d = np.ldexp(f, 62).astype(np.int64) - int(w * 2.0 ** 62)
    return (int((d >> 32).sum()) << 32) + int((d & 0xffffffff).sum())


@pytest.mark.parametrize("force", [0.0, 1e-6])
@pytest.mark.parametrize("tau", [0.55, 0.65, 0.9, 2.0])
def test_mass_and_momentum_keep_their_mean(tau, force):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    n = (128, 128, 128)
    nc = n[0] * n[1] * n[2]
    c, w = dps.lattice()
    rng = np.random.default_rng(11)
    u = 0.02 * rng.uniform(-1, 1, (3, nc))
    rho, uu = rng.uniform(0.98, 1.02, nc), 1.5 * (u ** 2).sum(0)
    f = np.empty((19, nc))
    for q in range(19):
        cu = c[q] @ u
        f[q] = w[q] * rho * (1 + 3 * cu + 4.5 * cu ** 2 - uu) * (1 + 1e-3 * rng.standard_normal(nc))
    dom = dps.Domain(n, (1, 1, 1), tau, "f64")
    dom.write_pdfs(f)
    fpf = force * rng.standard_normal((3, nc))
    if force:
        dom.write_fields(eps_f=rng.uniform(0.4, 1.0, nc), f_pf=fpf)
    # (the force sums: 2^21 terms of 1e-6 round to less than 1e-16 of 1e-3 a component)
    gain = np.ldexp(np.array([fpf[a].sum() for a in range(3)]), 62)
    for step in (1, 2):
        s0 = [exact_sum(f[q], w[q]) for q in range(19)]
        dom.collide_stream(1)
        f = dom.read_pdfs()
        d = [exact_sum(f[q], w[q]) - s0[q] for q in range(19)]
        mean = lambda x: float(x) * 2.0 ** -62 / nc
        assert abs(mean(sum(d))) <= 6 * 1.7e-17 / nc ** 0.5, step
        for a in range(3):
            j = sum(int(c[q][a]) * d[q] for q in range(19))
            assert abs(mean(j - int(gain[a]))) <= 6 * 4.1e-18 / nc ** 0.5, (step, a)
    dom.close()
