"""The workloads this library is timed on, through its public entry points.

A case is one use of the library: flocks of the k-nearest, Voronoi and metric
rules in 2D and 3D from the smallest system (launch latency) to the largest,
a batch of replicas, the tissue model and the allocation-free neighbor lists.
A pass of a flock restores a state (``set_state``, as teacher forcing and
checkpoint resume do), advances it ``steps`` time steps and reads the new
state back into device tensors, so every pass on the same state does the same
work.  A pass of the replica batch goes on from where the last one ended, as
a parameter sweep does, and reads every replica's order parameter and state.

``exact`` restates the path in 64-bit torch (integer distances, FP64
headings): k nearest and metric neighbors from a cell list or all pairs, 2D
Voronoi neighbors by clipping each bisector against the nearest particles.
It has no value for 3D Voronoi cells, for the replica batch and for large
clustered systems (all pairs would take too long).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2103_10239_gb300 import vk
from paper_2103_10239_gb300 import workloads as W

DEV = "cuda"


def listed():
    return [
        # a small flock run for a while and watched through its order parameter: launches and latency
        dict(name="flock_2k", kind="knn", dim=2, dist="uniform", n=2048, k=7, frac_bits=16, noise="angular",
             steps=50, eta=0.3, fov=False),
        # an ordinary flock of odd size, more neighbors, Eq. (2)'s own (vectorial) noise
        dict(name="flock_50k_k16", kind="knn", dim=2, dist="uniform", n=50021, k=16, frac_bits=16,
             noise="vectorial", steps=10, eta=0.3, fov=False),
        # the large clustered flock (256 Gaussian clusters on a background, density 1)
        dict(name="flock_clustered_4m", kind="knn", dim=2, dist="clustered", n=1 << 22, k=7, frac_bits=20,
             noise="angular", steps=10, eta=0.2, fov=False),
        # the same shape with particles that only see the half-plane ahead
        dict(name="flock_view_1m", kind="knn", dim=2, dist="clustered", n=1 << 20, k=7, frac_bits=20,
             noise="angular", steps=4, eta=0.2, fov=True),
        # a parameter sweep: 512 independent flocks of 1024 to 65536 particles in one batch, CUDA graph of 10 steps
        dict(name="replicas_512", kind="batch", replicas=512, lo=1024, hi=65536, k=7, steps=20, size_seed=1004),
        # a flock in 3D
        dict(name="flock3d_1m", kind="knn", dim=3, dist="uniform", n=1 << 20, k=7, frac_bits=20,
             noise="vectorial", steps=5, eta=0.2, fov=False),
        # the original Vicsek rule on the large clustered flock (hundreds of neighbors in the cores)
        dict(name="metric_4m", kind="metric", dim=2, dist="clustered", n=1 << 22, r0=1.0, frac_bits=20,
             noise="angular", steps=3, eta=0.2),
        # Voronoi flocks: uniform beside a stretched lattice, at low noise; and a large uniform one
        dict(name="voronoi_mixed_65k", kind="voronoi", dim=2, dist="mixed", n=65536, frac_bits=16, density=1.0,
             noise="angular", steps=10, eta=0.1, rebuild=False),
        dict(name="voronoi_1m", kind="voronoi", dim=2, dist="uniform", n=1 << 20, frac_bits=20, density=2.0,
             noise="angular", steps=2, eta=0.25, rebuild=False),
        dict(name="voronoi3d_262k", kind="voronoi", dim=3, dist="uniform", n=1 << 18, frac_bits=15, density=1.0,
             noise="vectorial", steps=1, eta=0.2, rebuild=False),
        # tissue model: areas, perimeters, energy and forces of a million cells, into host arrays
        dict(name="tissue_1m", kind="tissue", n=1 << 20, KA=1.0, KP=1.0, A0=1.0, P0=3.8),
        # neighbor lists for a caller that may not allocate (largest size of that entry point)
        dict(name="lists_65k", kind="lists", n=65536, k=7, frac_bits=16),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["knn", "knn", "knn", "knn3", "metric", "metric3", "voronoi", "voronoi", "voronoi3", "batch",
                       "tissue", "lists"])
    if kind == "knn":
        n = _log_int(rng, 256, 1 << 22)
        k = rng.choice([7, 7, rng.randint(1, 16), rng.randint(1, 32)])
        fov = rng.random() < 0.2
        if fov:
            n, k = min(n, 1 << 20), min(k, 7)
        dist = "clustered" if n >= 16384 and rng.random() < 0.5 else "uniform"
        k = k if n <= 1 << 18 else min(k, 16) if n <= 1 << 20 else 7
        steps = 50 if n <= 8192 else 10 if not fov else 4
        return dict(kind="knn", dim=2, dist=dist, n=n, k=k, frac_bits=rng.choice([16, 20]) if n <= 1 << 22 else 16,
                    noise=rng.choice(["angular", "angular", "vectorial"]), steps=steps,
                    eta=round(rng.uniform(0.05, 0.6), 3), fov=fov)
    if kind == "knn3":
        n = _log_int(rng, 512, 1 << 20)
        return dict(kind="knn", dim=3, dist="uniform", n=n, k=rng.choice([7, 7, 4, 14]) if n < 1 << 19 else 7,
                    frac_bits=rng.choice([16, 20]), noise="vectorial", steps=20 if n <= 8192 else 5,
                    eta=round(rng.uniform(0.05, 0.6), 3), fov=False)
    if kind == "metric":
        n = _log_int(rng, 1024, 1 << 22)
        dist = "clustered" if n >= 16384 and rng.random() < 0.5 else "uniform"
        return dict(kind="metric", dim=2, dist=dist, n=n,
                    r0=round(rng.uniform(0.5, 1.0 if dist == "clustered" else 2.0), 3),
                    frac_bits=rng.choice([16, 20]), noise=rng.choice(["angular", "vectorial"]),
                    steps=20 if n <= 8192 else 3, eta=round(rng.uniform(0.05, 0.6), 3))
    if kind == "metric3":
        n = _log_int(rng, 1024, 1 << 20)
        return dict(kind="metric", dim=3, dist="uniform", n=n, r0=round(rng.uniform(0.7, 1.5), 3), frac_bits=16,
                    noise="vectorial", steps=20 if n <= 8192 else 3, eta=round(rng.uniform(0.05, 0.6), 3))
    if kind == "voronoi":
        n = _log_int(rng, 128, 1 << 20)
        return dict(kind="voronoi", dim=2, dist="uniform", n=n, frac_bits=16,
                    density=round(rng.uniform(1.0, 2.0), 3), noise=rng.choice(["angular", "vectorial"]),
                    steps=20 if n <= 8192 else 5 if n <= 1 << 18 else 2, eta=round(rng.uniform(0.05, 0.5), 3),
                    rebuild=rng.random() < 0.25)
    if kind == "voronoi3":
        n = _log_int(rng, 256, 1 << 18)
        return dict(kind="voronoi", dim=3, dist="uniform", n=n, frac_bits=15, density=1.0, noise="vectorial",
                    steps=5 if n <= 8192 else 1, eta=round(rng.uniform(0.05, 0.5), 3), rebuild=False)
    if kind == "batch":
        return dict(kind="batch", replicas=_log_int(rng, 4, 400), lo=1024, hi=rng.choice([4096, 16384, 65536]),
                    k=rng.choice([7, 7, rng.randint(3, 10)]), steps=rng.choice([10, 20]),
                    size_seed=rng.randrange(1 << 20))
    if kind == "tissue":
        return dict(kind="tissue", n=_log_int(rng, 128, 1 << 20), KA=1.0, KP=round(rng.uniform(0.1, 2.0), 3), A0=1.0,
                    P0=round(rng.uniform(3.3, 4.0), 3))
    return dict(kind="lists", n=_log_int(rng, 64, 65536), k=rng.choice([7, 7, rng.randint(1, 32)]),
                frac_bits=rng.choice([16, 20]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _flock(c, seed):
    """The workload of one system: positions, headings, box and run parameters."""
    s = 1 << 20 | seed & 0x3FFFFFFF
    n, kind = c["n"], c["kind"]
    if kind in ("tissue", "lists"):
        return W.uniform_system(n, math.sqrt(n), c.get("frac_bits", 16), 2, s, rule="voronoi" if kind == "tissue" else "knn",
                                k=c.get("k", 0))
    rule, k = kind, c.get("k", 0)
    if c["dist"] == "mixed":
        return W.voronoi_mixed(eta=c["eta"], seed=s)
    if c["dist"] == "clustered":
        w = W.clustered_large(n=n, k=k, seed=s)
        if c["frac_bits"] != w.frac_bits:  # the same points on a coarser grid
            box = W.box_q_for(math.sqrt(n), c["frac_bits"])
            w.pos_q = np.minimum(w.pos_q >> (w.frac_bits - c["frac_bits"]), box - 1).astype(np.int32)
            w.box_q, w.frac_bits = (box, box), c["frac_bits"]
    else:
        length = (n / c.get("density", 1.0)) ** (1.0 / c["dim"])
        w = W.uniform_system(n, length, c["frac_bits"], c["dim"], s)
    w.rule, w.k, w.noise, w.eta = rule, k, c["noise"], c["eta"]
    w.v0, w.dt, w.seed = 0.3 if kind == "voronoi" and c["dim"] == 2 else 0.5, 1.0, 1
    return w


def _options(c):
    if c["kind"] == "metric":
        return {"r0": c["r0"]}
    if c["kind"] == "voronoi":
        return {"voronoi_rebuild": 1} if c["rebuild"] else {}
    return {"fov": 1, "fov_cos": 0.0} if c.get("fov") else {}


def _sizes(c):
    return W.replica_sizes(c["replicas"], c["lo"], c["hi"], seed=c["size_seed"])


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        sizes = _sizes(c)
        ws = W.replica_batch(k=c["k"], seed=seed & 0x3FFFFFFF, sizes=sizes)
        sim = vk.batch_from_workloads(ws, phi_capacity=64)
        sim.set_graph_steps(10)
        sim.step(20)  # a sweep that is under way
        sim.sync()
        n = int(sizes.sum())
        return dict(case=c, sim=sim, ends=np.concatenate([[0], np.cumsum(sizes)]).tolist(),
                    pos=torch.empty((n, 2), dtype=torch.int32, device=DEV),
                    dirs=torch.empty((n, 2), dtype=torch.float32, device=DEV))
    w = _flock(c, seed)
    if kind == "lists":
        return dict(case=c, box=w.box_q, pos=torch.from_numpy(w.pos_q).to(DEV),
                    ids=torch.empty((w.n, c["k"]), dtype=torch.int32, device=DEV))
    sim = vk.from_workload(w, **({} if kind == "tissue" else _options(c)))
    if kind == "tissue":
        return dict(case=c, sim=sim)
    pos, dirs = torch.from_numpy(w.pos_q).to(DEV), torch.from_numpy(w.dir).to(DEV)
    return dict(case=c, sim=sim, pos0=pos, dirs0=dirs, pos=torch.empty_like(pos), dirs=torch.empty_like(dirs))


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "lists":
        vk.knn_lists_noalloc(state["pos"], state["box"], c["frac_bits"], c["k"], state["ids"])
        return state["ids"]
    sim = state["sim"]
    if kind == "tissue":
        area, perimeter, energy, force = sim.tissue(c["KA"], c["KP"], c["A0"], c["P0"])
        return {"area": area, "perimeter": perimeter, "energy": energy, "force": force}
    if kind == "batch":
        sim.step(c["steps"])
        ends, phi = state["ends"], []
        for r in range(c["replicas"]):
            phi.append(sim.order_parameter(r, c["steps"]))
            sim.get_state_into(r, state["pos"][ends[r]:ends[r + 1]], state["dirs"][ends[r]:ends[r + 1]])
        return {"pos": state["pos"], "dirs": state["dirs"], "phi": np.stack(phi)}
    sim.set_state(state["pos0"], state["dirs0"], step=0)
    sim.step(c["steps"])
    phi = sim.order_parameter(0, c["steps"])
    sim.get_state_into(0, state["pos"], state["dirs"])
    return {"pos": state["pos"], "dirs": state["dirs"], "phi": phi}


def work(case):
    """Every step reads and writes each particle's position and heading (the
    definition of the step's roofline); the operations are one distance and
    one heading sum per neighbor and the update."""
    c = dict(case)
    kind = c["kind"]
    if kind == "lists":
        return {"bytes": c["n"] * (8 + 4 * c["k"]), "flops": c["n"] * c["k"] * 5}
    if kind == "tissue":
        return {"bytes": c["n"] * (8 + 32) + 8, "flops": c["n"] * 6 * 150}
    if kind == "batch":
        n = int(_sizes(c).sum())
        return {"bytes": c["steps"] * n * 32, "flops": c["steps"] * n * (c["k"] * 9 + 60)}
    d = c["dim"]
    m = c["k"] if kind == "knn" else 6 if d == 2 else 15.5
    if kind == "metric":
        m = math.pi * c["r0"] ** 2 if d == 2 else 4.19 * c["r0"] ** 3
        if c["dist"] == "clustered":  # 80 % of the particles in 256 Gaussian clusters of width 4
            m = 0.2 * m + 0.8 * (m + 0.8 * c["n"] / 256 * (1.0 - math.exp(-c["r0"] ** 2 / 64.0)))
    return {"bytes": c["steps"] * c["n"] * 16 * d, "flops": c["steps"] * c["n"] * (m * (3 * d + d) + 60)}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def _wrap(d, box):
    """Differences into (-L/2, L/2] (int64, last axis = box axes)."""
    d = torch.where(2 * d > box, d - box, d)
    return torch.where(2 * d <= -box, d + box, d)


def _offsets(pos, box, rows, cols):
    return _wrap(pos[cols] - pos[rows][:, None, :], box)


def _pairs_all(pos, box, rows, pick):
    """pick(rows, cols, offsets, D) over all particles, in chunks of rows."""
    n = pos.shape[0]
    step = max(1, (1 << 27) // n)
    cols = torch.arange(n, device=pos.device)
    for a in range(0, rows.shape[0], step):
        r = rows[a:a + step]
        off = _wrap(pos[None, :, :] - pos[r][:, None, :], box)
        dist = (off * off).sum(-1)
        dist[torch.arange(r.shape[0], device=pos.device), r] = 1 << 62
        pick(r, cols.expand(r.shape[0], n), off, dist)


def _pairs_cells(pos, box, per_cell, pick):
    """pick(rows, cols, offsets, D, width) over the 3^d cells around each particle (missing entries at D = 2^62);
    False when the box has fewer than three cells along an axis."""
    n, d = pos.shape
    dev = pos.device
    nc = [max(1, int(float(box[a]) / (float(torch.prod(box.double())) * per_cell / n) ** (1.0 / d))) for a in range(d)]
    if min(nc) < 3:
        return False
    nct = torch.tensor(nc, device=dev)
    cell = pos * nct // box
    width = int((box // nct).min())
    lin = cell[:, 0]
    for a in range(1, d):
        lin = lin * nc[a] + cell[:, a]
    order = torch.argsort(lin)
    total = math.prod(nc)
    count = torch.bincount(lin, minlength=total)
    first = torch.cumsum(count, 0) - count
    most = int(count.max())
    table = torch.full((total, most), -1, dtype=torch.int64, device=dev)
    sl = lin[order]
    table[sl, torch.arange(n, device=dev) - first[sl]] = order
    shifts = torch.cartesian_prod(*[torch.arange(-1, 2, device=dev)] * d)
    step = max(1, (1 << 25) // (most * 3 ** d))
    for a in range(0, n, step):
        r = order[a:a + step]
        near = (cell[r][:, None, :] + shifts) % nct
        g = near[..., 0]
        for ax in range(1, d):
            g = g * nc[ax] + near[..., ax]
        cols = table[g].reshape(r.shape[0], -1)
        off = _offsets(pos, box, r, cols.clamp(min=0))
        dist = (off * off).sum(-1)
        dist[(cols < 0) | (cols == r[:, None])] = 1 << 62
        pick(r, cols, off, dist, width)
    return True


def _nearest(pos, box, k, clustered, view=None):
    """The k nearest of every particle (columns by distance) and their squared distances; view = headings: only
    particles ahead count (short rows end in -1)."""
    n = pos.shape[0]
    ids = torch.full((n, k), -1, dtype=torch.int64, device=pos.device)
    dk = torch.full((n, k), 1 << 62, dtype=torch.int64, device=pos.device)
    sure = torch.zeros(n, dtype=torch.bool, device=pos.device)

    def pick(r, cols, off, dist, width=None):
        if view is not None:
            ahead = (off.double() * view[r][:, None, :]).sum(-1) >= 0
            dist = torch.where(ahead, dist, torch.full_like(dist, 1 << 62))
        v, at = torch.topk(dist, min(k, dist.shape[1]), dim=1, largest=False, sorted=True)
        got = torch.gather(cols, 1, at)
        got[v >= 1 << 62] = -1
        ids[r, :v.shape[1]], dk[r, :v.shape[1]] = got, v
        sure[r] = True if width is None else v[:, -1].double().sqrt() <= width

    if not clustered and view is None:
        _pairs_cells(pos, box, k * (0.75 if pos.shape[1] == 2 else 0.8) + 2, pick)
    left = torch.nonzero(~sure).flatten()
    if left.shape[0]:
        _pairs_all(pos, box, left, pick)
    return ids, dk


def _voronoi_lists(pos, box, k=28):
    """2D Voronoi neighbors of every particle as edges (i, j, l0, l1): j's edge of cell i ends at the circumcenters
    of (i, j, l0) and (i, j, l1).  Each bisector is clipped by the k nearest particles; a cell is final once the
    k-th lies beyond twice its farthest vertex, the others are repeated with four times as many."""
    n = pos.shape[0]
    todo = torch.arange(n, device=pos.device)
    parts = []
    while todo.shape[0]:
        k = min(k, n - 1)
        if todo.shape[0] == n:
            ids, dk = _nearest(pos, box, k, False)
        else:
            ids = torch.empty((todo.shape[0], k), dtype=torch.int64, device=pos.device)
            dk = torch.empty_like(ids)
            place = torch.full((n,), -1, dtype=torch.int64, device=pos.device)
            place[todo] = torch.arange(todo.shape[0], device=pos.device)

            def pick(r, cols, off, dist):
                v, at = torch.topk(dist, k, dim=1, largest=False, sorted=True)
                ids[place[r]], dk[place[r]] = at, v

            _pairs_all(pos, box, todo, pick)
        again = []
        step = max(1, (1 << 26) // (k * k))
        for a in range(0, todo.shape[0], step):
            r, c = todo[a:a + step], ids[a:a + step]
            q = _offsets(pos, box, r, c).double()
            q2 = (q * q).sum(-1)
            perp = torch.stack([-q[..., 1], q[..., 0]], -1)
            # point q_j / 2 + t perp_j is nearer to the particle than to l iff t * slope <= room
            slope = 2.0 * torch.einsum("rlx,rjx->rjl", q, perp)
            room = q2[:, None, :] - torch.einsum("rlx,rjx->rjl", q, q)
            t = room / slope
            inf = torch.full_like(t, math.inf)
            hi, l1 = torch.where(slope > 0, t, inf).min(-1)
            lo, l0 = torch.where(slope < 0, t, -inf).max(-1)
            dead = ((slope == 0) & (room < 0)).any(-1)
            edge = (hi > lo) & ~dead
            far = torch.maximum(hi.abs(), lo.abs())
            r2 = torch.where(edge, q2 * (0.25 + far * far), torch.zeros_like(q2)).amax(-1)
            final = (4.0 * r2 <= dk[a:a + step, -1].double()) | (k == n - 1)
            again.append(r[~final])
            row, j = torch.nonzero(edge & final[:, None], as_tuple=True)
            parts.append(torch.stack([r[row], c[row, j], c[row, l0[row, j]], c[row, l1[row, j]]], 1))
        todo = torch.cat(again)
        if k == n - 1:
            break
        k *= 4
    return torch.cat(parts)


def _philox(ids, step, replica, key):
    """Words 0 and 1 of Philox4x32-10 for counters (id, step, replica, 0)."""
    mask = 0xFFFFFFFF

    def mul(m, x):
        lo, hi = m * (x & 0xFFFF), m * (x >> 16)
        mid = hi + (lo >> 16)
        return mid >> 16 & mask, ((mid & 0xFFFF) << 16 | lo & 0xFFFF) & mask

    c = [ids & mask, torch.full_like(ids, step), torch.full_like(ids, replica), torch.zeros_like(ids)]
    k0, k1 = key & mask, key >> 32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return [(x >> 8).double() * 2.0 ** -24 for x in c[:2]]


def _update(w, pos, box, dirs, total, m, step):
    n, d = dirs.shape
    u, u1 = _philox(torch.arange(n, device=pos.device), step, 0, w.seed)
    eta, s = float(np.float32(w.eta)), float(np.float32(w.v0 * w.dt)) * 2.0 ** w.frac_bits
    if w.noise == "angular":
        zero = (total == 0).all(-1, keepdim=True)
        base = torch.where(zero, dirs, total)
        th = torch.atan2(base[:, 1], base[:, 0]) + eta * (u - 0.5)
        new = torch.stack([th.cos(), th.sin()], 1)
    else:
        ang = 2.0 * math.pi * u
        if d == 2:
            xi = torch.stack([ang.cos(), ang.sin()], 1)
        else:
            z = 2.0 * u1 - 1.0
            r = (1.0 - z * z).clamp(min=0).sqrt()
            xi = torch.stack([r * ang.cos(), r * ang.sin(), z], 1)
        v = eta * xi + total / m.clamp(min=1).double()[:, None]
        norm = (v * v).sum(-1, keepdim=True).sqrt()
        new = torch.where(norm == 0, dirs, v / norm)
    return (pos + torch.round(s * dirs).to(torch.int64)) % box, new


def _exact_step(c, w, pos, box, dirs, step):
    n = pos.shape[0]
    clustered = c["dist"] == "clustered"
    total, m = torch.zeros_like(dirs), torch.zeros(n, dtype=torch.int64, device=pos.device)
    if c["kind"] == "knn":
        ids, _ = _nearest(pos, box, c["k"], clustered, dirs if c["fov"] else None)
        total = (dirs[ids.clamp(min=0)] * (ids >= 0)[..., None]).sum(1)
        m = (ids >= 0).sum(1)
    elif c["kind"] == "metric":
        r2 = int(np.rint(np.float64(np.float32(c["r0"])) * 2.0 ** w.frac_bits)) ** 2

        def pick(r, cols, off, dist, width=None):
            near = dist <= r2
            m[r] = near.sum(1)
            row, at = torch.nonzero(near, as_tuple=True)
            total[r] = torch.zeros_like(total[r]).index_add_(0, row, dirs[cols[row, at]])

        per = 1.05 * n * float(r2) ** (w.dim / 2) / float(torch.prod(box.double())) + 1
        if clustered or not _pairs_cells(pos, box, per, pick):
            _pairs_all(pos, box, torch.arange(n, device=pos.device), pick)
    else:
        e = _voronoi_lists(pos, box)
        total.index_add_(0, e[:, 0], dirs[e[:, 1]])
        m.index_add_(0, e[:, 0], torch.ones_like(e[:, 0]))
    return _update(w, pos, box, dirs, total, m, step)


def _exact_tissue(c, w, pos, box):
    e = _voronoi_lists(pos, box)
    unit = 2.0 ** -w.frac_bits
    i = e[:, 0]
    at = pos.double() * unit
    at.requires_grad_(True)
    size = box.double() * unit

    def rel(j):  # offset from particle i, differentiable
        d = at[j] - at[i]
        return d - (size * torch.round(d.detach() / size))

    def center(a, b):
        cross = 2.0 * (a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0])
        a2, b2 = (a * a).sum(-1), (b * b).sum(-1)
        return torch.stack([(b[:, 1] * a2 - a[:, 1] * b2) / cross, (a[:, 0] * b2 - b[:, 0] * a2) / cross], 1)

    h0, h1 = center(rel(e[:, 1]), rel(e[:, 2])), center(rel(e[:, 1]), rel(e[:, 3]))
    zero = torch.zeros(pos.shape[0], dtype=torch.float64, device=pos.device)
    area = zero.index_add(0, i, 0.5 * (h0[:, 0] * h1[:, 1] - h0[:, 1] * h1[:, 0]))
    perim = zero.index_add(0, i, ((h1 - h0) ** 2).sum(-1).sqrt())
    energy = (c["KA"] * (area - c["A0"]) ** 2 + c["KP"] * (perim - c["P0"]) ** 2).sum()
    force, = torch.autograd.grad(-energy, at)
    return {"area": area.detach().cpu().numpy(), "perimeter": perim.detach().cpu().numpy(),
            "energy": float(energy.detach()), "force": force.cpu().numpy()}


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind in ("batch", "lists") or kind == "voronoi" and c["dim"] == 3:
        return None
    slow = c.get("dist") == "clustered" or c.get("fov")
    if slow and c["n"] > 1 << 17 or c["n"] < 256:
        return None
    w = _flock(c, seed)
    pos, box = torch.from_numpy(w.pos_q).to(DEV).long(), torch.tensor(w.box_q, device=DEV, dtype=torch.int64)
    if kind == "tissue":
        return _exact_tissue(c, w, pos, box)
    dirs, phi = torch.from_numpy(w.dir).to(DEV).double(), []
    for step in range(c["steps"]):
        pos, dirs = _exact_step(c, w, pos, box, dirs, step)
        phi.append(float(dirs.sum(0).square().sum().sqrt()) / c["n"])
    return {"pos": None, "dirs": dirs, "phi": np.array(phi)}
