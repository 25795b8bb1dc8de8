"""2D kNN: long lists of particles whose square cannot decide (close distances,
squares too wide or too small), with the squares that are scanned for them."""
import numpy as np
import pytest

from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flock(pos, box, k):
    return W.Workload(name="handed", dim=2, pos_q=np.ascontiguousarray(pos, np.int32), dir=W.random_dirs(len(pos)), theta=None,
                      box_q=box, frac_bits=16, rule="knn", k=k, v0=0.0, eta=0.3)


def _lattice(shake):
    pos, box = W.square_lattice(200, 1 << 16)
    return (pos + np.random.default_rng(3).integers(-shake, shake + 1, pos.shape)) % box[0], box


# distances that a thread cannot order stay so: one square by a thread, one by a group, none in between
@pytest.mark.parametrize("k", [6, 7, 14])
def test_close_distances_are_not_scanned_again(k):
    with vk.from_workload(_flock(*_lattice(0), k)) as sim:
        sim.step(1)  # (the first squares are guessed)
        sim.set_profiling(True, True)
        sim.step(1)
        c = sim.search_counters()
        assert c["updates"] == 40000 and c["rf_walk_tie"] == 40000
        assert c["runs_or_squares"] == 2 * c["updates"]


# every kind of long list gives what the general search gives: close distances, squares with few hits, a strip that
# they span
@pytest.mark.parametrize("kind", ["lattice", "shaken", "few", "strip"])
@pytest.mark.parametrize("k", [7, 12])
def test_long_lists_as_the_general_search(kind, k):
    rng = np.random.default_rng(k)
    if kind == "strip":
        w = _flock(np.stack([rng.integers(0, 1 << 26, 40000), rng.integers(0, 2000, 40000)], 1), (1 << 26, 2000), k)
    elif kind == "few":
        w = _flock(rng.integers(0, 1 << 24, (40000, 2)), (1 << 24, 1 << 24), k)
    else:
        w = _flock(*_lattice(kind == "shaken"), k)
    got = []
    for search in (0, 1):
        with vk.from_workload(w, knn_search=search, search_halo=0.5 if kind == "few" else 0.0) as sim:
            lists = sim.neighbors()[1]
            sim.step(3)
            got.append((lists, sim.neighbors()[1]) + sim.state()[:2])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
