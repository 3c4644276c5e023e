"""A caller's allocator that aligns to 8 or 16 bytes: the domain runs in its memory with
the bits of a run in aligned memory, and gives every block back once."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("shift", [8, 16])
def test_allocator_of_small_alignment(form, shift, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps, workloads
    n, per = (14, 12, 16), (1, 0, 1)
    pr = workloads.random_particles(n, per, 60, seed=3)
    alloc, free = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete
    held = {}

    def shifted_alloc(nbytes, *a):
        p = alloc(nbytes + shift, *a)
        held[p + shift] = p
        return p + shift

    out = []
    for odd in (False, True):
        if odd:
            monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", shifted_alloc)
            monkeypatch.setattr(torch.cuda, "caching_allocator_delete", lambda p: free(held.pop(p)))
        dom = dps.Domain(n, per, 0.7, form, max_particles=60)
        dom.add_particles(pr["x"], pr["d"], pr["rho_p"], u=pr["u"], w=pr["w"])
        dom.set_closure(g=(0, 0, -1e-4), T_c=4.0, h_c=0.5, n_int=2, n_dem=4, skin=0.9, lift=1)
        dom.step(3)
        out.append({**dom.read_particles(), **dom.read_fields(("ubar", "f_pf"))})
        assert bool(held) == odd
        dom.close()
    assert not held
    for k, v in out[0].items():
        assert np.isfinite(v).all() and np.array_equal(v, out[1][k]), k
