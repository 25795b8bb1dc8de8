"""Creating and closing sims: the pinned host blocks that closed sims leave to
the next ones."""
import time
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flock(n=500, seed=1):
    return W.uniform_system(n, n ** 0.5, 14, 2, input_seed=seed, rule="knn", k=7, v0=0.5, eta=0.3)


# about 370 us; two pinned allocations of its own made it 670
def test_a_small_sim_costs_no_pinned_allocation():
    w = _flock()
    vk.from_workload(w).close()
    us = []
    for _ in range(60):
        t = time.perf_counter()
        vk.from_workload(w).close()
        us.append((time.perf_counter() - t) * 1e6)
    assert min(us) < 560


# more sims at once than blocks are kept, opened, read and closed by several threads: each reads its own values
def test_sims_on_threads_read_their_own_values():
    want = {}
    for seed in range(6):
        with vk.from_workload(_flock(seed=seed)) as sim:
            sim.step(20)
            want[seed] = sim.order_parameter()
    assert len({v.tobytes() for v in want.values()}) == 6

    def work(i):
        sims = [vk.from_workload(_flock(seed=(i + j) % 6)) for j in range(5)]
        for _ in range(4):
            for s in sims:
                s.step(5)
        ok = [np.array_equal(s.order_parameter(), want[(i + j) % 6]) for j, s in enumerate(sims)]
        for s in sims:
            s.sync()
            s.close()
        return all(ok)

    with ThreadPoolExecutor(6) as pool:
        assert all(pool.map(work, range(24)))
