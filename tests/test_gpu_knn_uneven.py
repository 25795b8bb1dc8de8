"""2D kNN where one particle's search could hold up all others: clusters with
particles far outside."""
import numpy as np
import pytest
import torch

import oracle
from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W
from parity import check_step

pytestmark = pytest.mark.gpu


def _cluster(n, sigma, L, at=0.5):
    rng = np.random.default_rng(n)
    return np.ascontiguousarray(rng.normal(at * L, sigma * L, (n, 2)).astype(np.int64) % L, np.int32)


def _flock(pos, L, k):
    return W.Workload(name="uneven", dim=2, pos_q=pos, dir=W.random_dirs(len(pos)), theta=None, box_q=(L, L),
                      frac_bits=12, rule="knn", k=k, v0=0.5, eta=0.3)


def _time(pos, L, k):
    out = torch.empty((len(pos), k), dtype=torch.int32, device="cuda")
    p = torch.from_numpy(pos).cuda()
    ms = []
    for _ in range(15):
        t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        t[0].record()
        vk.knn_lists_noalloc(p, (L, L), 12, k, out)
        t[1].record()
        torch.cuda.synchronize()
        ms.append(t[0].elapsed_time(t[1]))
    return sorted(ms)[7]


# first radii are guessed from the density around a particle: outside a cluster they may hold all of it.  One
# thread needs 20 times as long for such a square as all lists of a uniform system take; with its share limited (40 us
# of about 130 at 1024 particles) and the rest left to groups, no system takes many times as long as another
@pytest.mark.parametrize("k", [7, 32])
def test_no_particle_holds_up_all_others(k):
    n, L = 65536, 1 << 24
    even = np.ascontiguousarray(np.random.default_rng(1).integers(0, L, (n, 2)), np.int32)
    assert _time(_cluster(n, 0.02, L), L, k) < 6 * _time(even, L, k)


# steps and lists of such systems, with and without hints, the cluster in the middle and across the corner
@pytest.mark.parametrize("k", [7, 12, 16, 32])
@pytest.mark.parametrize("n,sigma,at", [(3000, 0.002, 0.5), (6000, 0.02, 0.0), (6000, 0.1, 0.5)])
def test_uneven_lists(n, sigma, at, k):
    L = 1 << 24
    pos = _cluster(n, sigma, L, at)
    w = _flock(pos, L, k)
    with vk.from_workload(w) as sim:
        for _ in range(2):
            check_step(sim, w, w.rule)
    out = torch.empty((n, k), dtype=torch.int32, device="cuda")
    vk.knn_lists_noalloc(torch.from_numpy(pos).cuda(), (L, L), 12, k, out)
    assert np.array_equal(out.cpu().numpy(), oracle.knn(pos, (L, L), k))
