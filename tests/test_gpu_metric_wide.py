"""2D metric rule: rectangles wider than half a period, on one axis or both."""
import numpy as np
import pytest

from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W
from parity import check_step
from test_gpu_rules import metric_lists, r0q_of

pytestmark = pytest.mark.gpu


# one axis covered whole and the other not, both a little below and above half a period and a period, a coarse cell
# met twice by a narrow rectangle
@pytest.mark.parametrize("box,r0", [((65536, 4096), 1.5), ((4096, 65536), 3.0), ((65536, 20000), 2.2), ((65536, 65536), 1.9),
                                    ((65536, 65536), 3.2), ((65536, 65536), 3.9), ((65537, 65535), 6.1), ((65536, 65536), 7.9)])
@pytest.mark.parametrize("n,occ", [(65, 0.0), (900, 0.0), (900, 4.0), (900, 5000.0)])
def test_wide_rectangles(box, r0, n, occ):
    rng = np.random.default_rng(n)
    pos = np.stack([rng.integers(0, b, n) for b in box], 1)
    w = W.Workload(name="wide", dim=2, pos_q=np.ascontiguousarray(pos, np.int32), dir=W.random_dirs(n), theta=None,
                   box_q=box, frac_bits=12, rule="metric", k=0, v0=0.5, eta=0.3)
    with vk.from_workload(w, r0=r0, cell_occupancy=occ) as sim:
        for _ in range(2):
            check_step(sim, w, w.rule, lists=metric_lists(box, r0q_of(r0, 12)))


# squares of 0.32 to 0.48 of the box's edge: the rectangles of cells of a sixth to an eighth of it hold well below all
@pytest.mark.parametrize("n,share", [(2000, 0.16), (2000, 0.2), (20000, 0.238)])
def test_wide_rectangles_do_not_take_the_whole_box(n, share):
    w = W.uniform_system(n, n ** 0.5, 16, 2, input_seed=n, rule="metric", k=0, v0=0.5, eta=0.3)
    with vk.from_workload(w, r0=share * n ** 0.5) as sim:
        sim.set_profiling(True, True)
        sim.step(1)
        assert sim.search_stats()["mean_candidates"] < 0.6 * n
