"""GPU parity of the kernels' routes at the sizes where they change: list
sizes the 2D and 3D searches are compiled for, squares that hold more hits
than a thread buffers, particles handed on from one kernel to the next (few
and many), rectangles of the metric rule across the period, Voronoi cells
around the edge and face counts at which a builder hands a cell on.  Lists and
positions are integers and compared element by element; headings within the
1e-5 rad of every teacher-forced step."""
import numpy as np
import pytest

import oracle
from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W
from parity import angle_between, check_step
from test_gpu_rules import metric_lists, r0q_of

pytestmark = pytest.mark.gpu


def _flock(pos, box, bits, dim, **kw):
    return W.Workload(name="routes", dim=dim, pos_q=np.ascontiguousarray(pos, np.int32),
                      dir=W.random_dirs(pos.shape[0], dim=dim), theta=None, box_q=box, frac_bits=bits,
                      noise="vectorial" if dim == 3 else "angular", **kw)


def _check(w, steps=2, lists=None, **kw):
    with vk.from_workload(w, **kw) as sim:
        for _ in range(steps):
            check_step(sim, w, w.rule, lists=lists)


# ------------------------------------------------------------------ k nearest

# one below, at and one above every compiled list size (7, 11, 16 | 32 in 2D, 7, 16 | 32 in 3D), the whole
# system as neighbors, and the general search alone
@pytest.mark.parametrize("search", [0, 1])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("k", [1, 6, 7, 8, 11, 12, 16, 17, 31, 32])
def test_knn_list_sizes(dim, k, search):
    for n in (k + 1, 641):
        w = W.uniform_system(n, max(3.0, n ** (1.0 / dim)), 14, dim, input_seed=10 * k + dim, rule="knn", k=k, v0=0.5,
                             eta=0.3, noise="vectorial" if dim == 3 else "angular")
        _check(w, knn_search=search)


# boxes that no power of two divides, long ones, one cell wide, and the largest coordinates
@pytest.mark.parametrize("box", [(1000003, 77777), (4096, 1 << 20), (1 << 31, 1 << 31), ((1 << 31) - 1, 3 << 20),
                                 (65537, 65535)])
@pytest.mark.parametrize("n,k", [(130, 7), (1500, 12)])
def test_knn_boxes(box, n, k):
    rng = np.random.default_rng(n + k)
    pos = np.stack([rng.integers(0, b, n) for b in box], 1)
    _check(_flock(pos, box, 10, 2, rule="knn", k=k, v0=0.5, eta=0.3))


# hints of a sparse state meet a dense one (squares of thousands of hits: full columns) and the reverse
# (squares of none: handed on); 40,000 particles make the list long enough for the kernel of second squares
@pytest.mark.parametrize("dim,n,k", [(2, 3000, 7), (2, 3000, 16), (2, 40000, 7), (3, 3000, 7), (3, 3000, 20)])
def test_knn_stale_hints(dim, n, k):
    rng = np.random.default_rng(n + k)
    L = 1 << 20
    wide = rng.integers(0, L, (n, dim))
    tight = (rng.normal(L / 2, L / 400, (n, dim)).astype(np.int64)) % L
    query = np.sort(rng.choice(n, 500, replace=False))
    d = W.random_dirs(n, dim=dim)
    w = _flock(wide, (L,) * dim, 16, dim, rule="knn", k=k, v0=0.5, eta=0.3)
    states = []
    for search in (0, 1):  # the general search takes no hints
        with vk.from_workload(w, knn_search=search) as sim:
            for pos in (tight, wide, tight):
                sim.step(1)
                sim.set_state(np.ascontiguousarray(pos, np.int32), d, step=1)
                sim.step(1)
                states.append(sim.state()[:2])
        with vk.from_workload(w, knn_search=search) as sim:
            sim.step(1)
            sim.set_state(np.ascontiguousarray(tight, np.int32), d, step=1)
            ids = sim.neighbors()[1].reshape(-1, k)
            assert np.array_equal(ids[query], oracle.knn(np.ascontiguousarray(tight, np.int32), w.box_q, k,
                                                         query=query))
    for a, b in zip(states[:3], states[3:]):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


# distances that FP32 keys cannot order: a fine lattice shaken by one unit, and coincident particles
@pytest.mark.parametrize("dim,m", [(2, 40), (3, 11)])
def test_knn_near_ties(dim, m):
    rng = np.random.default_rng(dim)
    a = 1 << 20
    grid = np.stack(np.meshgrid(*[np.arange(m)] * dim, indexing="ij"), -1).reshape(-1, dim) * a
    pos = (grid + rng.integers(-1, 2, grid.shape)) % (m * a)
    pos[1::97] = pos[::97][:pos[1::97].shape[0]]
    for k in (5, 8, 14):
        _check(_flock(pos, (m * a,) * dim, 20, dim, rule="knn", k=k, v0=0.0, eta=0.3))


# -------------------------------------------------------------------- metric

# warps whose particles lie in several coarse cells, rectangles across the period, just below and above half a
# period, one particle more and less than a warp and a block
@pytest.mark.parametrize("n,box,r0", [(31, (40960, 40960), 3.0), (33, (40960, 40960), 9.9), (129, (1000003, 33333), 2.5),
                                      (700, (65536, 65536), 7.0), (700, (65536, 65536), 15.5), (700, (65536, 65536), 16.5),
                                      (2000, (1 << 31, 1 << 31), 90000.0)])
@pytest.mark.parametrize("occ", [4.0, 256.0])
def test_metric_2d_rectangles(n, box, r0, occ):
    rng = np.random.default_rng(n)
    pos = np.stack([rng.integers(0, b, n) for b in box], 1)
    pos[: n // 3] = (rng.normal(0, 400, (n // 3, 2)).astype(np.int64)) % np.array(box)  # a cluster on the corner
    w = _flock(pos, box, 12, 2, rule="metric", k=0, v0=0.5, eta=0.3)
    _check(w, lists=metric_lists(box, r0q_of(r0, 12)), r0=r0, cell_occupancy=occ)


# cubes inside one cell, over several, across the period, and too wide for the row walk
@pytest.mark.parametrize("r0", [0.05, 1.0, 2.4, 2.6, 6.0])
def test_metric_3d_cubes(r0):
    rng = np.random.default_rng(3)
    box = (10240, 11003, 40000)
    pos = np.stack([rng.integers(0, b, 900) for b in box], 1)
    w = _flock(pos, box, 10, 3, rule="metric", k=0, v0=0.5, eta=0.3)
    _check(w, lists=metric_lists(box, r0q_of(r0, 10)), r0=r0)


# ------------------------------------------------------------------- Voronoi

def _ring(m, dim, L=1 << 15):
    """A particle alone in a void with m others at nearly one distance (its cell has m edges or faces), more outside."""
    rng = np.random.default_rng(m)
    c, r = L / 2, 0.22 * L
    if dim == 2:
        ang = np.arange(m) * (2 * np.pi / m)
        u = np.stack([np.cos(ang), np.sin(ang)], 1)
    else:  # a spiral on the sphere: about evenly spread
        z = 1 - (2 * np.arange(m) + 1) / m
        phi = np.arange(m) * np.pi * (3 - np.sqrt(5.0))
        s = np.sqrt(1 - z * z)
        u = np.stack([s * np.cos(phi), s * np.sin(phi), z], 1)
    shell = c + r * u + rng.uniform(-1, 1, (m, dim))
    out = rng.uniform(0, L, (400, dim))
    out = out[np.linalg.norm(out - c, axis=1) > 1.25 * r]
    pos = np.concatenate([[[c + 3] * dim], shell, out]).astype(np.int64)
    return pos, (L,) * dim


# eight lanes hold 8 edges each once and 16 twice; more go to the warp kernel
@pytest.mark.parametrize("m", [7, 8, 9, 10, 14, 15, 16, 17, 24])
def test_voronoi_2d_edge_counts(m):
    pos, box = _ring(m, 2)
    w = _flock(pos, box, 9, 2, rule="voronoi", k=0, v0=0.3, eta=0.2)
    with vk.from_workload(w) as sim:
        off, _ = sim.neighbors()
        assert off[1] - off[0] == m
        area, perimeter, energy, force = sim.tissue(1.0, 1.0, 1.0, 3.8)
        oa, op, oe, of = oracle.tissue(w.pos_q, box, 9, 1.0, 1.0, 1.0, 3.8)
        assert np.allclose(area, oa, rtol=1e-9, atol=0) and np.allclose(perimeter, op, rtol=1e-9, atol=0)
        assert energy == pytest.approx(oe, rel=1e-9)
        assert np.abs(force - of).max() <= 1e-7 * np.abs(of).max()
    for rebuild in (0, 1):
        _check(w, steps=3, voronoi_rebuild=rebuild)


# one, two and eight rounds of cells per warp: the same headings whatever the grouping
@pytest.mark.parametrize("n", [1, 4, 5, 127, 129, 60001, 240001])
def test_voronoi_2d_rounds(n):
    w = W.uniform_system(n, max(n, 2) ** 0.5, 16, 2, input_seed=n, rule="voronoi", k=0, v0=0.3, eta=0.2)
    if n < 1000:
        _check(w)
        return
    with vk.from_workload(w) as sim:
        pos, d, _, t = sim.state()
        sim.step(1)
        pos1, d1, _, _ = sim.state()
    off, ids = oracle.voronoi(pos, w.box_q)
    op, od, _ = oracle.vicsek_step(pos, d, w.box_q, off, ids, frac_bits=w.frac_bits, v0=w.v0, dt=w.dt, eta=w.eta,
                                   seed=w.seed, step=t)
    assert np.array_equal(pos1, op)
    assert angle_between(d1, od).max() <= 1e-5


# the small cell holds 64 planes and 128 vertices (about 66 faces), the large one twice that
@pytest.mark.parametrize("m", [12, 30, 33, 58, 62, 66, 90, 100])
def test_voronoi_3d_face_counts(m):
    pos, box = _ring(m, 3)
    _check(_flock(pos, box, 9, 3, rule="voronoi", k=0, v0=0.3, eta=0.2))


# a batch of sizes that leave ragged ends in every grouping of cells
def test_voronoi_3d_batch_ends():
    ws = [W.uniform_system(n, n ** (1.0 / 3.0), 15, 3, input_seed=70 + n, rule="voronoi", k=0, v0=0.5, eta=0.3,
                           noise="vectorial") for n in (15, 257, 16, 300, 33)]
    with vk.batch_from_workloads(ws) as sim:
        for r, w in enumerate(ws):
            off, ids = sim.neighbors(r)
            want = oracle.voronoi3(w.pos_q, w.box_q)
            assert np.array_equal(off, want[0]) and np.array_equal(ids, want[1])
        pos0, d0 = zip(*[sim.state(r)[:2] for r in range(len(ws))])
        sim.step(1)
        for r, w in enumerate(ws):
            pos1, d1, _, _ = sim.state(r)
            off, ids = oracle.voronoi3(pos0[r], w.box_q)
            op, od, _ = oracle.vicsek_step(pos0[r], d0[r], w.box_q, off, ids, frac_bits=w.frac_bits, v0=w.v0, dt=w.dt,
                                           eta=w.eta, seed=w.seed, step=0, replica=r, noise=w.noise)
            assert np.array_equal(pos1, op) and angle_between(d1, od).max() <= 1e-5
