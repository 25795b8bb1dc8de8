"""2D Voronoi: the neighbors that wide cells keep from the last step (seeds) are
used, and lists and states stay exact whatever state they come from."""
import numpy as np
import pytest

import oracle
from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W
from parity import check_step

pytestmark = pytest.mark.gpu


def _work(rebuild):
    with vk.from_workload(W.voronoi_mixed(eta=0.1, seed=3), voronoi_rebuild=rebuild) as sim:
        sim.step(80)
        sim.set_profiling(True, True)
        sim.step(5)
        return sim.search_stats()


# a flock with grown voids: the cells beside them are bounded by their seeds, so they meet fewer particles and
# fewer of them need the warp kernel than without
def test_seeds_spare_candidates_beside_voids():
    reuse, rebuild = _work(0), _work(1)
    assert reuse["mean_candidates"] < 0.9 * rebuild["mean_candidates"]
    assert reuse["split_fraction"] < 0.9 * rebuild["split_fraction"]


def _void(n, L, seed):
    rng = np.random.default_rng(seed)
    p = rng.integers(0, L, (2 * n, 2))
    return p[np.hypot(*(p - L // 2).T) > 0.35 * L][:n]


# seeds of a state with a void meet another void, a uniform state, a mirrored one and one with coincident particles
@pytest.mark.parametrize("n", [300, 2500])
def test_seeds_of_another_state(n):
    L = 1 << 18
    pos = _void(n, L, n)
    w = W.Workload(name="reuse", dim=2, pos_q=np.ascontiguousarray(pos, np.int32), dir=W.random_dirs(n), theta=None,
                   box_q=(L, L), frac_bits=12, rule="voronoi", k=0, v0=0.3, eta=0.2)
    twins = _void(n, L, 7)
    twins[1::50] = twins[::50][:twins[1::50].shape[0]]
    others = (_void(n, L, n + 1), np.random.default_rng(5).integers(0, L, (n, 2)), L - 1 - pos, twins)
    with vk.from_workload(w) as sim:
        check_step(sim, w, w.rule)
        for other in others:
            for p in (other, pos):
                sim.set_state(np.ascontiguousarray(p, np.int32), w.dir, step=3)
                check_step(sim, w, w.rule)
                check_step(sim, w, w.rule)
        sim.set_state(np.ascontiguousarray(others[0], np.int32), w.dir, step=3)
        area, perimeter, energy, _ = sim.tissue(1.0, 1.0, 1.0, 3.8)
        want = oracle.tissue(np.ascontiguousarray(others[0], np.int32), (L, L), 12, 1.0, 1.0, 1.0, 3.8)
        assert np.allclose(area, want[0], rtol=1e-9, atol=0) and np.allclose(perimeter, want[1], rtol=1e-9, atol=0)
