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
@pytest.mark.parametrize("dim,n,rule,passes", [(2, 1000, "voronoi", 2), (2, 10000, "voronoi", 2), (3, 5000, "knn", 1),
                                               (3, 1000, "knn", 1)])
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


# 3D: groups alone (small systems), cubes by threads and the groups for what they leave: ordinary, close distances, a
# cluster whose first radii are far off; before steps and after
@pytest.mark.parametrize("kind", ["uniform", "lattice", "cluster"])
@pytest.mark.parametrize("m,k", [(6, 7), (33, 7), (33, 13), (33, 32)])
def test_knn3_lists_of_every_route(kind, m, k):
    rng = np.random.default_rng(m + k)
    n, L = m ** 3, m << 14
    if kind == "lattice":
        pos = W.cubic_lattice("sc", m, 1 << 14)[0]
    elif kind == "cluster":
        pos = rng.normal(L / 2, L / 100, (n, 3)).astype(np.int64) % L
    else:
        pos = rng.integers(0, L, (n, 3))
    w = W.Workload(name="export3", dim=3, pos_q=np.ascontiguousarray(pos, np.int32), dir=W.random_dirs(n, dim=3), theta=None,
                   box_q=(L,) * 3, frac_bits=14, rule="knn", k=k, v0=0.02, eta=0.3, noise="vectorial")
    query = np.sort(rng.choice(n, min(n, 400), replace=False))
    with vk.from_workload(w) as sim:
        for steps in (0, 2):
            sim.step(steps)
            ids = sim.neighbors()[1].reshape(-1, k)
            assert np.array_equal(ids[query], oracle.knn(sim.state()[0], w.box_q, k, query=query))
