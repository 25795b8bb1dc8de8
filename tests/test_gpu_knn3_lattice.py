"""3D kNN of lattices and of particles at equal distances, large enough for the
search by one thread per particle."""
import numpy as np
import pytest

import oracle
from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flock(pos, box, k):
    return W.Workload(name="lattice3", dim=3, pos_q=np.ascontiguousarray(pos, np.int32), dir=W.random_dirs(len(pos), dim=3),
                      theta=None, box_q=tuple(box), frac_bits=14, rule="knn", k=k, v0=0.0, eta=0.3, noise="vectorial")


def _positions(kind):
    rng = np.random.default_rng(2)
    if kind == "coincident":
        p = rng.integers(0, 1 << 19, (6000, 3))
        return p[rng.integers(0, 6000, 35000)], (1 << 19,) * 3
    pos, box = W.cubic_lattice(kind.split("-")[0], {"sc": 33, "bcc": 26, "fcc": 21}[kind.split("-")[0]], 1 << 14)
    if kind.endswith("shaken"):
        pos = (pos + rng.integers(-1, 2, pos.shape)) % np.array(box)
    return pos, box


# threads order equal and nearly equal distances exactly: lists as the oracle's, steps as the general search's
@pytest.mark.parametrize("kind", ["sc", "bcc", "fcc", "sc-shaken", "fcc-shaken", "coincident"])
@pytest.mark.parametrize("k", [4, 7, 8, 13, 16])
def test_equal_distances(kind, k):
    pos, box = _positions(kind)
    w = _flock(pos, box, k)
    query = np.arange(0, len(pos), 97)
    got = []
    for search in (0, 1):
        with vk.from_workload(w, knn_search=search) as sim:
            sim.step(2)
            ids = sim.neighbors()[1].reshape(-1, k)
            assert np.array_equal(ids[query], oracle.knn(w.pos_q, box, k, query=query))
            got.append(sim.state()[1])
    assert np.array_equal(got[0], got[1])


# a cube of half-width 1.2 sqrt(2) lattice spacings meets three or four cells of 1.6 an axis: nine rows of slots or more;
# a particle left to a group counts its cubes alone, one or two
def test_lattice_particles_are_not_handed_on():
    pos, box = _positions("sc")
    with vk.from_workload(_flock(pos, box, 7)) as sim:
        sim.step(1)
        sim.set_profiling(True, True)
        sim.step(1)
        c = sim.search_counters()
        assert c["updates"] == len(pos) and c["runs_or_squares"] > 6 * len(pos)
