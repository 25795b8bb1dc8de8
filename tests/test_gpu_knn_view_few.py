"""Field of view that holds fewer than k particles: the search of the next step
begins with the whole box instead of growing to it again."""
import pytest

from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W
from parity import check_step
from test_gpu_rules import fov_lists

pytestmark = pytest.mark.gpu


# at 0.45 % of the directions in view, 600 particles (5000) hold about 3 (22) of the 7 (31) wanted; hardly any holds all
@pytest.mark.parametrize("n,k", [(600, 7), (5000, 31)])
def test_short_views(n, k):
    w = W.uniform_system(n, n ** 0.5, 16, 2, input_seed=n, rule="knn", k=k, v0=0.05, eta=0.3)
    cos = 0.9999
    with vk.from_workload(w, fov=1, fov_cos=cos) as sim:
        for _ in range(3):
            check_step(sim, w, w.rule, lists=fov_lists(w.box_q, k, cos))
        sim.set_profiling(True, True)
        sim.step(1)
        c = sim.search_counters()
        assert c["updates"] == n and c["runs_or_squares"] < 2 * n
