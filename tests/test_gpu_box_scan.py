"""The cell offsets of a box (scan tiles of 4096 cells): one tile, a last tile of
any size, several tiles, and more tiles than the tile kernel sums directly, against a
histogram of the cells; again after steps, whose sorts count the cells anew."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def offsets(x, n):
    c = np.floor(x).astype(np.int64)
    key = c[:, 0] + n[0] * (c[:, 1] + n[1] * c[:, 2])
    return np.concatenate([[0], np.cumsum(np.bincount(key, minlength=n[0] * n[1] * n[2]))])


@pytest.mark.parametrize("n,count", [((5, 3, 4), 9), ((16, 16, 16), 700), ((17, 16, 15), 900), ((19, 17, 13), 800),
                                     ((64, 33, 31), 5000), ((257, 256, 256), 4000)])
def test_cell_offsets(n, count):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    rng = np.random.default_rng(count)
    x = rng.random((count, 3)) * n
    dom = dps.Domain(n, (1, 1, 1), 0.7, "f16s", max_particles=count)
    dom.add_particles(x, 0.3, 2.5, u=0.01 * rng.standard_normal((count, 3)))
    dom.set_closure(n_int=2, n_dem=1, contact=0, lubrication=0, drag=0, pressure=0, added_mass=0, skin=0.5)
    dom.prepare()
    start, order = dom.read_cell_list()
    assert np.array_equal(start, offsets(x, n))
    assert np.array_equal(np.sort(order), np.arange(count))
    dom.step(2)
    start, order = dom.read_cell_list()
    assert np.array_equal(start, offsets(dom.read_particles()["x"], n))
    assert np.array_equal(np.sort(order), np.arange(count))
    dom.close()
