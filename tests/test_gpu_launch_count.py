"""launches_per_step before a step, after it, and after a change of the closure: the number
the phases of the step then count, for every route of the step."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = {  # form, box, particles
    "one_sphere": ("f64", (16, 16, 20), 1),
    "few": ("f64", (24, 24, 24), 100),
    "many": ("f64", (24, 24, 24), 400),
    "fluid": ("f64", (8, 8, 8), 0),
    "mixed_solo": ("f32", (16, 16, 16), 20),
    "mixed_few": ("f32", (24, 24, 24), 400),
    "mixed_many": ("f32", (64, 64, 64), 40000),
    "half_few": ("f16s", (24, 24, 24), 300),
    "many_cells": ("f16s", (257, 256, 256), 10),
}


@pytest.mark.parametrize("name", list(CASES))
def test_count_is_that_of_the_next_step(name):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    form, n, k = CASES[name]
    dom = dps.Domain(n, (1, 1, 1), 0.6, form, max_particles=max(k, 1))
    if k:
        dom.add_particles(np.random.default_rng(0).random((k, 3)) * n, 0.3, 2.5)
    dom.set_timing(True)
    for kw in (dict(n_int=2, n_dem=5), dict(n_int=3, n_dem=4, lift=1), dict(n_int=1, n_dem=5, eilers=1)):
        dom.set_closure(g=(0, 0, 0), fb_mode=0, contact=0, lubrication=0, skin=0.5, **kw)
        before = dom.launches_per_step()
        dom.get_timing()
        dom.step(1)
        dom.collect_timing()
        count = sum(v["launches"] for v in dom.get_timing().values())
        assert before == count
        assert dom.launches_per_step() == count
    dom.close()


def test_count_of_a_batch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    for form in ("f64", "f32"):
        b = dps.Batch(form)
        for j, (n, k) in enumerate((((16, 16, 16), 30), ((24, 20, 16), 300), ((40, 40, 40), 9000))):
            i = b.add_box(n, (1, 1, 1), 0.6, max_particles=k)
            b.add_particles(i, np.random.default_rng(j).random((k, 3)) * n, np.full(k, 0.3), np.full(k, 2.5))
            b.set_closure(i, g=(0, 0, 0), fb_mode=0, contact=0, lubrication=0, n_int=2, n_dem=4, skin=0.5,
                          smagorinsky=j % 2)
            before = b.launches_per_step()
            b.step(1)
            assert b.launches_per_step() == before, (form, j)
        b.close()
