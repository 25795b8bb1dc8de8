"""The warp builder of 3D Voronoi cells (its own clipping and linking; it shares
the predicates with the serial builder that the host test compiles) on the
degenerate and order-sensitive configurations of that test: lists and one step
against the oracle, with the particles in several orders and in cells of several
sizes, which change the order in which sites are clipped."""
import numpy as np
import pytest

import oracle
from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W
from parity import angle_between

pytestmark = pytest.mark.gpu


def _grid():
    return np.unique(np.random.default_rng(10).integers(0, 8, (150, 3)) * 16, axis=0), (128, 128, 128)


def _jittered():
    m, sp = 8, 1 << 12
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) * sp
    return (g + np.random.default_rng(11).integers(-2, 3, g.shape)) % (m * sp), (m * sp,) * 3


def _uniform(n, box, seed):
    return np.random.default_rng(seed).integers(0, box, (n, 3)), box


CASES = {
    "grid": _grid, "jittered": _jittered,
    "sc": lambda: W.cubic_lattice("sc", 4, 1 << 10, offset_q=(1, 2, 3)),
    "bcc": lambda: W.cubic_lattice("bcc", 4, 1 << 10, offset_q=(1, 2, 3)),
    "fcc": lambda: W.cubic_lattice("fcc", 4, 1 << 10, offset_q=(1, 2, 3)),
    "anisotropic": lambda: _uniform(200, (500, 900, 3000), 9),
    "large": lambda: _uniform(600, (1 << 23,) * 3, 8),
    "tiny": lambda: _uniform(8, (500,) * 3, 4),
}


@pytest.mark.parametrize("occ", [0.3, 0.0, 40.0])
@pytest.mark.parametrize("case", sorted(CASES))
def test_cells_in_any_order(case, occ):
    pos, box = CASES[case]()
    off, ids = oracle.voronoi3(np.ascontiguousarray(pos, np.int32), box)
    n = len(pos)
    for seed in range(3):
        perm = np.random.default_rng(seed).permutation(n) if seed else np.arange(n)
        place = np.argsort(perm)  # old number -> new
        q = np.ascontiguousarray(pos[perm], np.int32)
        d = W.random_dirs(n, dim=3, seed=seed)
        with vk.Sim.create(q, d, box, 10, rule="voronoi", noise="vectorial", v0=0.5, eta=0.3, cell_occupancy=occ) as sim:
            goff, gids = sim.neighbors()
            for i in range(n):
                assert np.array_equal(gids[goff[i]:goff[i + 1]], np.sort(place[ids[off[perm[i]]:off[perm[i] + 1]]]))
            sim.step(1)
            pos1, d1, _, _ = sim.state()
        op, od, _ = oracle.vicsek_step(q, d, box, goff, gids, frac_bits=10, v0=0.5, dt=1.0, eta=0.3, seed=1, step=0,
                                       noise="vectorial")
        assert np.array_equal(pos1, op) and angle_between(d1, od).max() <= 1e-5
