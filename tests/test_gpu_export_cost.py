"""Neighbor lists cost about what the searches of a step cost, and are exact by
every route of the exporting kernels."""
import numpy as np
import pytest

import oracle
from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cost(sim):
    """ms of a list export and of a step's search from the same state, over some states."""
    ms = []
    for _ in range(8):
        sim.set_profiling(True)
        sim.neighbors()  # (two exports: the count, then the lists)
        sim.step(1)
        p = sim.profile()
        ms.append((p["export"][0] / 2, p["search_update"][0]))
    return np.median(ms, axis=0)


# every pass searches once; 0.1 ms for the copies to the host and the waits between
@pytest.mark.parametrize("dim,n,rule,passes", [(2, 1000, "voronoi", 2), (2, 10000, "voronoi", 2)])
def test_export_costs_its_searches(dim, n, rule, passes):
    w = W.uniform_system(n, n ** (1.0 / dim), 15, dim, input_seed=n, rule=rule, k=7, v0=0.3, eta=0.3,
                         noise="vectorial" if dim == 3 else "angular")
    with vk.from_workload(w) as sim:
        sim.step(5)
        export, search = _cost(sim)
        assert export < passes * 1.5 * search + 0.1


# ordinary cells, cells that a warp builds (a cluster in a void), coincident particles, after steps (seeds) and before
@pytest.mark.parametrize("n", [5, 131, 2000])
def test_voronoi_lists_of_every_route(n):
    rng = np.random.default_rng(n)
    L = 1 << 20
    pos = np.concatenate([rng.integers(0, L, (n // 3, 2)), rng.normal(L / 2, L / 200, (n - n // 3, 2)).astype(np.int64) % L])
    if n > 100:
        pos[5::40] = pos[4::40][: pos[5::40].shape[0]]
    w = W.Workload(name="export", dim=2, pos_q=np.ascontiguousarray(pos, np.int32), dir=W.random_dirs(n), theta=None,
                   box_q=(L, L), frac_bits=12, rule="voronoi", k=0, v0=0.3, eta=0.2)
    with vk.from_workload(w) as sim:
        for _ in range(3):
            want = oracle.voronoi(sim.state()[0], (L, L))
            got = sim.neighbors()
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
            sim.step(4)
