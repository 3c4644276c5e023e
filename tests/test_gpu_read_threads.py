"""Several domains read back at once: the helper threads of all calls together are at most
seven, and every read returns its own particles."""
import os
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_concurrent_reads_share_the_helpers():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_00336_gb300 import dps
    n, count, readers = (64, 64, 64), 300000, 5
    rng = np.random.default_rng(6)
    xs, doms = [], []
    for _ in range(readers):
        x = rng.random((count, 3)) * n
        dom = dps.Domain(n, (1, 1, 1), 0.7, "f64", max_particles=count)
        dom.add_particles(x, 0.3, 2.5)
        dom.read_particles()
        xs.append(x)
        doms.append(dom)
    start, bad = threading.Barrier(readers + 1), []

    def read(k):
        start.wait()
        for _ in range(12):
            if not np.array_equal(doms[k].read_particles()["x"], xs[k]):
                bad.append(k)

    team = [threading.Thread(target=read, args=(k,)) for k in range(readers)]
    for t in team:
        t.start()
    before = len(os.listdir("/proc/self/task"))
    start.wait()
    most = before
    while any(t.is_alive() for t in team):
        most = max(most, len(os.listdir("/proc/self/task")))
    for t in team:
        t.join()
    for dom in doms:
        dom.close()
    assert not bad
    assert most - before <= 7
