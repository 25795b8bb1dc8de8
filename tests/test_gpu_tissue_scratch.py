"""Device memory that the tissue model keeps: packed rows of the cells' edges."""
import numpy as np
import pytest
import torch

import oracle
from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# rows of 32 entries of slot and offset (384 bytes), the row's length, area, perimeter, and 33 bytes of outputs a
# particle are what a system of a given size has always had to find room for
def test_scratch_per_particle():
    n = 1 << 20
    with vk.from_workload(W.uniform_system(64, 8.0, 16, 2, input_seed=3, rule="voronoi", k=0)) as sim:
        sim.tissue(1.0, 1.0, 1.0, 3.8)  # the kernels' stack, which the context keeps whatever the system's size
    w = W.uniform_system(n, 1024.0, 20, 2, input_seed=3, rule="voronoi", k=0, v0=0.3, eta=0.2)
    with vk.from_workload(w) as sim:
        sim.sync()
        before = torch.cuda.mem_get_info()[0]
        sim.tissue(1.0, 1.0, 1.0, 3.8)
        assert before - torch.cuda.mem_get_info()[0] <= 440 * n


# cells of very different edge counts side by side: rows that straddle everything, several replicas on one scratch
@pytest.mark.parametrize("n", [3, 5, 33, 500])
def test_rows_of_uneven_cells(n):
    rng = np.random.default_rng(n)
    L = 1 << 16
    ws = []
    for r in range(3):
        pos = rng.integers(0, L, (n + r, 2))
        ang = np.sort(rng.uniform(0, 2 * np.pi, 14))
        ring = L / 2 + 0.3 * L * np.stack([np.cos(ang), np.sin(ang)], 1)
        if n > 20:  # one cell of up to 14 edges in a void
            pos = pos[np.hypot(*(pos - L / 2).T) > 0.36 * L]
            pos = np.concatenate([pos, ring.astype(np.int64), [[L // 2 + 5, L // 2 - 9]]])
        ws.append(W.Workload(name="rows", dim=2, pos_q=np.ascontiguousarray(pos, np.int32), dir=W.random_dirs(len(pos)),
                             theta=None, box_q=(L, L), frac_bits=12, rule="voronoi", k=0, v0=0.3, eta=0.2))
    with vk.batch_from_workloads(ws) as sim:
        for r in (0, 2, 1, 0):
            area, perimeter, energy, force = sim.tissue(1.0, 2.0, 1.5, 3.0, replica=r)
            oa, op, oe, of = oracle.tissue(ws[r].pos_q, (L, L), 12, 1.0, 2.0, 1.5, 3.0)
            assert np.allclose(area, oa, rtol=1e-9, atol=0) and np.allclose(perimeter, op, rtol=1e-9, atol=0)
            assert energy == pytest.approx(oe, rel=1e-9)
            assert np.abs(force - of).max() <= 1e-7 * np.abs(of).max()
