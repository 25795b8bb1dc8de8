"""An occupancy tuned for one kind of system is not taken for another whose default differs."""
import pytest

from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flock(n):
    return W.uniform_system(n, n ** 0.5, 14, 2, input_seed=n, rule="knn", k=7, v0=0.5, eta=0.3)


def _cells(make):
    with make() as sim:
        return sim.info().n_cells


# views against plain flocks, and replicas that are large together against one system of their size
@pytest.mark.parametrize("tuned,other", [
    (lambda: vk.from_workload(_flock(140000)), lambda: vk.from_workload(_flock(140000), fov=1, fov_cos=0.0)),
    (lambda: vk.from_workload(_flock(3000), fov=1, fov_cos=0.0), lambda: vk.from_workload(_flock(3000))),
    (lambda: vk.from_workload(_flock(3000)), lambda: vk.batch_from_workloads([_flock(3000)] * 48)),
])
def test_tuned_occupancy_stays_with_its_kind(tuned, other):
    vk.autotune_forget()
    try:
        before = _cells(other)
        with tuned() as sim:
            assert sim.autotune([9.0], trial_steps=1) == 9.0
            cells = sim.info().n_cells
        assert _cells(tuned) == cells  # its own kind starts from it
        assert _cells(other) == before
    finally:
        vk.autotune_forget()
