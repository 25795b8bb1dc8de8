"""Benchmark: particle-steps/s of the fused non-metric neighbor build + Vicsek
step (kNN, k=7) at N = 2^22 on one GB300, with the HBM-roofline fraction of
the dominant kernel, an end-to-end figure through the C ABI with host
buffers, and the CPU oracle timed on the host cores.

A "step" is one pass of the whole hot path: the kNN search fused with the
alignment/noise/advection update, the cell-count scan and the scatter into
cell-sorted order.

Usage:  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
Multi-GPU (torchrun): every rank runs its own independent replica of the
workload (replicas only, weak scaling); rank 0 prints the JSON line.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import re
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "particle-steps/s (neighbor build + Vicsek step), N=4M k=7, and % HBM roofline"
ALG_BYTES_PER_PARTICLE_STEP = 24  # pos int32x2 + heading fp32, read and written once
CSRC = os.path.join(ROOT, "paper_2103_10239_gb300", "csrc")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--n", type=int, default=1 << 22)
    ap.add_argument("--k", type=int, default=7)
    ap.add_argument("--layout", choices=["clustered", "uniform"], default="clustered")
    ap.add_argument("--e2e-steps", type=int, default=5)
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--voronoi3-kernel", type=int, choices=[0, 1], default=None,
                    help="voronoi3d scenario: passed to the library, where 0 and 1 are the same kernel")
    ap.add_argument("--scenario-n", type=int, default=0,
                    help="particles of the voronoi3d / knn3d scenario (0: the workload's default)")
    ap.add_argument("--occupancy", type=float, default=64.0,
                    help="coarse-grid occupancy (particles per cell) of the headline run; 64 is what the "
                         "library takes for a flock of this size when it is left to it")
    ap.add_argument("--search", choices=["radius", "walk"], default="radius",
                    help="2D kNN search: radius-first squares (default) or the general search of lane groups only")
    ap.add_argument("--halo", type=float, default=0.0,
                    help="radius-first search square half-width as a multiple of the previous k-th "
                         "distance (0: library default)")
    ap.add_argument("--no-replicas", action="store_true",
                    help="skip the replica-batch block of the headline line")
    ap.add_argument("--no-secondary", action="store_true",
                    help="skip the short secondary measurements (other rules and dimensions)")
    ap.add_argument("--replica-steps", type=int, default=10,
                    help="timed (and warm-up) steps of each arm of the replica-batch block")
    ap.add_argument("--autotune", action="store_true",
                    help="let the library's autotuner pick the occupancy on the warmed-up state instead")
    ap.add_argument("--scenario", choices=["headline", "replicas", "voronoi", "voronoi3d", "knn3d"], default="headline",
                    help="headline: the benchmark line; the others are secondary measurements")
    return ap.parse_args()


def workload(args, rank=0):
    from paper_2103_10239_gb300 import workloads as W
    if args.layout == "clustered":
        return W.clustered_large(n=args.n, k=args.k, seed=1003 + 100 * rank)
    return W.uniform_large(n=args.n, k=args.k, seed=1013 + 100 * rank)


def workload_config(w, args):
    return {"workload": w.name, "n": w.n, "rule": w.rule, "k": w.k, "dim": w.dim,
            "frac_bits": w.frac_bits, "box_q": int(w.box_q[0]), "density": round(w.density, 4),
            "v0": w.v0, "eta": w.eta, "layout": args.layout, "search": args.search,
            "l2": "flushed between timed steps (256 MiB write)"}


# ---------------------------------------------------------------------------
# clocks sampled during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.dev), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.t.join(timeout=2)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax), "reasons": sorted(reasons),
                "samples": len(sm)}


# ---------------------------------------------------------------------------
# roofline bookkeeping
# ---------------------------------------------------------------------------
def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        try:
            d = json.load(open(p))
            return float(d["hbm_gbs"]), "measured"
        except Exception:
            pass
    return 6800.0, "fallback"


def kernel_source_sha() -> str:
    """Hash of the sources the dominant kernel (knn2_box_step_kernel) is built from."""
    h = hashlib.sha256()
    for f in ("vk_internal.cuh", "vk_box2d.cuh", "vk_knn2d.cu"):
        h.update(open(os.path.join(CSRC, f), "rb").read())
    return h.hexdigest()[:16]


def recorded_traffic(workload_name: str, occupancy):
    """DRAM bytes per launch of the search+update kernel from the committed
    ncu summary, if it was taken on the current kernel sources, workload and
    coarse-grid occupancy."""
    p = os.path.join(ROOT, "profiles", "knn2_box_step_kernel_clustered4M.md")
    if not os.path.exists(p):
        return None
    txt = open(p).read()
    m_sha = re.search(r"source_sha256_16:\s*([0-9a-f]+)", txt)
    m_b = re.search(r"dram_bytes_per_launch_full_workload:\s*([0-9.e+]+)", txt)
    m_w = re.search(r"workload:\s*(\S+)", txt)
    if not (m_sha and m_b and m_w):
        return None
    if m_sha.group(1) != kernel_source_sha() or m_w.group(1) != workload_name:
        return None
    m_o = re.search(r"cell_occupancy:\s*([0-9.]+)", txt)
    if m_o is None or occupancy is None or float(m_o.group(1)) != float(occupancy):
        return None
    return float(m_b.group(1))


# ---------------------------------------------------------------------------
# CPU oracle baseline (the oracle as it stands, on the host cores)
# ---------------------------------------------------------------------------
def oracle_sample_rate(w, budget_s: float, min_q: int = 32, m_fixed=None, seed: int = 0):
    """Oracle particle-steps/s on a bounded sample: brute-force kNN of a
    random subset of particles over all N plus the FP64 update, scaled to
    the subset.  Without m_fixed the subset grows until the search takes
    about budget_s."""
    import oracle
    oracle.build()
    rng = np.random.default_rng(seed)
    # grow the sample until the brute-force search takes about the budget
    m = m_fixed or min_q
    while True:
        q = np.sort(rng.choice(w.n, m, replace=False)).astype(np.int64)
        t0 = time.perf_counter()
        nb = oracle.knn(w.pos_q, w.box_q, w.k, query=q)
        t_knn = time.perf_counter() - t0
        if m_fixed or t_knn >= 0.6 * budget_s or m >= w.n:
            break
        m = int(min(w.n, max(2 * m, m * 0.9 * budget_s / max(t_knn, 1e-6))))
    # the update of the sampled particles (run on a system made of them)
    off = np.arange(m + 1, dtype=np.int64) * w.k
    remap = np.full(w.n, -1, dtype=np.int64)
    remap[q] = np.arange(m)
    sub_ids = remap[nb.ravel()]
    sub_ids[sub_ids < 0] = 0  # neighbours outside the sample: any valid index (timing only)
    t0 = time.perf_counter()
    oracle.vicsek_step(w.pos_q[q], w.dir[q], w.box_q, off, sub_ids.astype(np.int32), frac_bits=w.frac_bits,
                       v0=w.v0, dt=w.dt, eta=w.eta, seed=w.seed, step=0, noise=w.noise)
    t_upd = time.perf_counter() - t0
    return m / (t_knn + t_upd), m, oracle.num_threads(), t_knn + t_upd


def scenario_cpu_baseline(w, budget_s: float) -> dict:
    """The oracle on the host cores for a secondary workload, on its initial
    state: a whole step (exact Delaunay triangulation of the periodic set,
    neighbor lists, FP64 update) for the Voronoi rule; a bounded sample for
    kNN."""
    import oracle
    oracle.build()
    if w.rule == "voronoi" and w.dim == 3:
        # the oracle builds each 3D cell independently: time a random sample
        m = min(w.n, 4096)
        q = np.sort(np.random.default_rng(7).choice(w.n, m, replace=False))
        t0 = time.perf_counter()
        oracle.voronoi3(w.pos_q, w.box_q, query=q)
        t = time.perf_counter() - t0
        return {"value": m / t, "unit": "particle-steps/s", "cores": oracle.num_threads(), "kind": "oracle",
                "sample": f"{m} random particles of the {w.n}-particle workload ({t:.1f} s): exact cell "
                          "clipping against all N particles (the FP64 update, a negligible share, not timed)"}
    if w.rule == "voronoi":
        t0 = time.perf_counter()
        off, ids = (oracle.voronoi3 if w.dim == 3 else oracle.voronoi)(w.pos_q, w.box_q)
        t_nb = time.perf_counter() - t0
        t0 = time.perf_counter()
        oracle.vicsek_step(w.pos_q, w.dir, w.box_q, off, ids, frac_bits=w.frac_bits, v0=w.v0, dt=w.dt,
                           eta=w.eta, seed=w.seed, step=0)
        t_upd = time.perf_counter() - t0
        return {"value": w.n / (t_nb + t_upd), "unit": "particle-steps/s", "cores": 1, "kind": "oracle",
                "sample": f"one whole step of all {w.n} particles ({t_nb + t_upd:.1f} s): "
                          + ("exact cell clipping on %d threads" % oracle.num_threads() if w.dim == 3
                             else "serial Bowyer-Watson triangulation")
                          + f" ({t_nb:.1f} s) + FP64 update on {oracle.num_threads()} threads"}
    rate, m, cores, secs = oracle_sample_rate(w, budget_s)
    return {"value": rate, "unit": "particle-steps/s", "cores": cores, "kind": "oracle",
            "sample": f"{m} random particles of the {w.n}-particle workload: brute-force kNN over all N "
                      f"+ FP64 update ({secs:.1f} s)"}


# ---------------------------------------------------------------------------
def run_reference(args, rank, world):
    if rank != 0:
        return
    w = workload(args)
    total_budget = 150.0
    per_step = total_budget / max(1, args.steps + args.warmup)
    _, m_used, _, _ = oracle_sample_rate(w, per_step)  # size the per-step sample once
    for i in range(args.warmup):
        oracle_sample_rate(w, per_step, m_fixed=m_used, seed=1 + i)
    times, parts = [], 0
    cores = 0
    for i in range(args.steps):
        rate, m, cores, secs = oracle_sample_rate(w, per_step, m_fixed=m_used, seed=100 + i)
        times.append(secs)
        parts += m
    value = parts / sum(times)
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "particle-steps/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * sum(times) / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "int64+f64", "data": "synthetic",
            "config": dict(workload_config(w, args), cell_occupancy=args.occupancy, l2_bytes=_l2_bytes()),
            "cpu_baseline": {"value": value, "unit": "particle-steps/s", "cores": cores, "kind": "oracle",
                             "sample": f"{m_used} random particles per step: brute-force kNN over all "
                                       f"{w.n} + FP64 update"},
            "e2e": {"value": value, "unit": "particle-steps/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def _l2_bytes():
    """L2 size of GPU 0, as the measured arm records it (None without a GPU)."""
    try:
        import torch
        if torch.cuda.is_available():
            return int(torch.cuda.get_device_properties(0).L2_cache_size)
    except Exception:
        pass
    return None


def reduce_job(dist, units: float, seconds: float, device):
    """Whole-job totals over the ranks: the units all ranks processed (sum)
    and the slowest rank's time (max).  Without a process group: unchanged."""
    if dist is None:
        return float(units), float(seconds)
    import torch
    u = torch.tensor([float(units)], dtype=torch.float64, device=device)
    t = torch.tensor([float(seconds)], dtype=torch.float64, device=device)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(u.item()), float(t.item())


def run_ours(args, rank, world, dist):
    import torch
    from paper_2103_10239_gb300 import vk
    from paper_2103_10239_gb300 import _build

    _build.build()
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    w = workload(args, rank)
    stream = torch.cuda.Stream(device=dev)
    torch.cuda.set_stream(stream)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    sim = vk.from_workload(w, stream=stream, cell_occupancy=args.occupancy,
                           knn_search=0 if args.search == "radius" else 1, search_halo=args.halo)
    sim.step(args.warmup)
    occupancy = args.occupancy
    if args.autotune:
        # the library's autotuner picks the coarse-grid occupancy on the
        # warmed-up state (state and step counter are restored afterwards)
        occupancy = sim.autotune([64.0, 128.0, 256.0, 512.0, 1024.0, 2048.0, 4096.0, 8192.0], trial_steps=2)
    torch.cuda.synchronize()
    sim.set_profiling(True)

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    clocks = ClockSampler(local)
    barrier()
    clocks.start()
    time.sleep(0.3)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    barrier()
    t_wall0 = time.perf_counter()
    for i in range(args.steps):
        flush.fill_(i & 0xFF)  # evict the state from L2 (outside the timed events)
        ev[i][0].record(stream)
        sim.step(1)
        ev[i][1].record(stream)
    barrier()
    t_wall = time.perf_counter() - t_wall0
    time.sleep(0.2)
    clk = clocks.stop()
    sim.sync()
    step_ms = [a.elapsed_time(b) for a, b in ev]
    total_ms = float(sum(step_ms))
    prof = sim.profile()
    sim.set_profiling(False)
    units, secs = reduce_job(dist, w.n * args.steps, total_ms * 1e-3, dev)
    ms_per_step = secs * 1e3 / args.steps
    value = units / secs

    # dominant kernel: the fused radius-first search + update of every
    # particle (phase search_update, one launch per step); the particles it
    # lists are finished in the search_deferred phase
    su_ms, su_launches = prof["search_update"]
    per_launch_ms = su_ms / max(1, su_launches)
    sd_ms = prof.get("search_deferred", (0.0, 0))[0]
    alg_bytes = ALG_BYTES_PER_PARTICLE_STEP * w.n
    peak, peak_kind = measured_peaks()
    achieved = alg_bytes / (per_launch_ms * 1e-3) / 1e9
    traffic = recorded_traffic(w.name, occupancy)

    # end to end through the C ABI with pinned host buffers
    e2e = None
    if True:  # every rank, so that the whole-job figure covers them all
        pos_h = torch.empty((w.n, 2), dtype=torch.int32, pin_memory=True)
        dir_h = torch.empty((w.n, 2), dtype=torch.float32, pin_memory=True)
        # the host-driven loop continues the simulation from its current state
        sim.get_state_into(0, pos_h, dir_h)
        phi_h = np.zeros(1, dtype=np.float64)
        barrier()
        t_e = []
        for i in range(args.e2e_steps + 1):
            t0 = time.perf_counter()
            sim.set_state(pos_h, dir_h)
            sim.step(1)
            sim.get_state_into(0, pos_h, dir_h)
            phi_h[0] = sim.order_parameter(max_values=1)[-1]
            t_e.append(time.perf_counter() - t0)
        t_e = t_e[1:]
        e_units, e_secs = reduce_job(dist, w.n * len(t_e), sum(t_e), dev)
        e2e = {"value": e_units / e_secs, "unit": "particle-steps/s",
               "h2d_bytes_per_step": int(w.n * 16), "d2h_bytes_per_step": int(w.n * 16 + 8),
               "note": "vk_set_state from pinned host + vk_step(1) + vk_get_state to pinned host + phi"}

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        rate, m, cores, secs = oracle_sample_rate(w, args.cpu_seconds)
        cpu = {"value": rate, "unit": "particle-steps/s", "cores": cores, "kind": "oracle",
               "sample": f"{m} random particles of the {w.n}-particle workload: brute-force kNN over "
                         f"all N + FP64 update ({secs:.1f} s)"}

    info = sim.info()
    sim.close()
    replicas = None
    if rank == 0 and world == 1 and not args.no_replicas:
        replicas = replica_block(stream, args.replica_steps)
    secondary = None
    if rank == 0 and world == 1 and not args.no_secondary:
        secondary = secondary_block(stream)
    if rank != 0:
        return
    phases = {k: {"ms_total": v[0], "launches": v[1]} for k, v in prof.items() if v[1]}
    line = {
        "metric": METRIC, "value": value, "unit": "particle-steps/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_per_step,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int64+f32",
        "data": "synthetic", "config": dict(workload_config(w, args), cell_occupancy=occupancy,
                                            l2_bytes=int(torch.cuda.get_device_properties(dev).L2_cache_size)),
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak, "traffic": traffic,
                     "kernel": "knn2_box_step_kernel (radius-first kNN search + align + advect)",
                     "alg_bytes_per_launch": alg_bytes, "peak_kind": f"{peak_kind} hbm_gbs (burst copy)",
                     "kernel_ms_per_launch": per_launch_ms,
                     "search_phase_ms_per_step": (su_ms + sd_ms) / args.steps},
        "step_roofline": {"achieved_gbs": alg_bytes / (ms_per_step * 1e-3) / 1e9,
                          "frac": alg_bytes / (ms_per_step * 1e-3) / 1e9 / peak,
                          "note": "24 B per particle-step over the whole step"},
        # secondary, labelled: the implementation's state with the heading as an
        # FP32 unit vector (pos 8 B + heading 8 B, read and written once)
        "roofline_float2_state": {"bytes_per_particle_step": 32,
                                  "achieved_gbs": 32 * w.n / (per_launch_ms * 1e-3) / 1e9,
                                  "frac": 32 * w.n / (per_launch_ms * 1e-3) / 1e9 / peak},
        "cpu_baseline": cpu, "e2e": e2e, "gpu_launches": int(info.kernels_per_step) * args.steps,
        "clocks": clk, "phases": phases, "wall_s_timed_region": t_wall, "replicas": replicas,
        "secondary": secondary,
    }
    print(json.dumps(line), flush=True)


def replica_block(stream, steps: int) -> dict:
    """The batched-replica pattern: 512 replicas (N_r log-uniform in
    [1024, 65536], k = 7, F = 16) stepped together (one launch per kernel,
    multi-step CUDA graph) against the same replicas as separate systems with
    one launch sequence each.  Both arms start from the same states, take the
    same number of warm-up steps, and evolve identically (each separate
    system draws its noise with its replica index)."""
    from paper_2103_10239_gb300 import vk
    from paper_2103_10239_gb300 import workloads as W
    ws = W.replica_batch()
    total = sum(w.n for w in ws)
    sim = vk.batch_from_workloads(ws, stream=stream)
    sim.set_graph_steps(steps)
    sim.step(steps)  # warm-up, also captures the graph
    ms_b = _timed(stream, lambda: sim.step(steps)) / steps
    pos_b, _, _, t_b = sim.state(300)
    sim.close()
    sims = [vk.from_workload(w, stream=stream, replica_offset=r) for r, w in enumerate(ws)]
    for x in sims:
        x.step(steps)  # the same warm-up

    def per_rep():
        for _ in range(steps):
            for x in sims:
                x.step(1)
    ms_p = _timed(stream, per_rep) / steps
    pos_p, _, _, t_p = sims[300].state()
    for x in sims:
        x.close()
    return {"metric": "particle-steps/s, 512 replicas in one launch per kernel + multi-step graph",
            "value": total / (ms_b * 1e-3), "unit": "particle-steps/s", "ms_per_step": ms_b,
            "per_replica_launches": {"value": total / (ms_p * 1e-3), "ms_per_step": ms_p},
            "speedup_vs_per_replica_launches": ms_p / ms_b,
            "warmup_steps_each_arm": steps, "timed_steps_each_arm": steps,
            "replica_300_identical_across_arms": bool(t_b == t_p and np.array_equal(pos_b, pos_p)),
            "config": {"workload": "512 replicas, N_r log-uniform [1024, 65536], density 1, k=7, F=16, "
                                   "eta 0.05-0.6", "n_total": total}}


def _rate(stream, sim, n: int, warmup: int, steps: int) -> dict:
    sim.step(warmup)
    ms = _timed(stream, lambda: sim.step(steps)) / steps
    return {"value": n / (ms * 1e-3), "unit": "particle-steps/s", "ms_per_step": ms, "warmup": warmup,
            "steps": steps}


def secondary_block(stream) -> dict:
    """Short measurements of the other rules and dimensions, each from its
    own seeded synthetic state, timed with CUDA events on the sim's stream
    over consecutive steps after a warm-up (inputs resident, no L2 flush
    between steps).  Labelled secondary: not the benchmark configuration."""
    from paper_2103_10239_gb300 import vk
    from paper_2103_10239_gb300 import workloads as W
    out = {}
    wv = W.voronoi_mixed(eta=0.1)
    for name, rebuild in (("voronoi_mixed65k_reuse", 0), ("voronoi_mixed65k_rebuild", 1)):
        with vk.from_workload(wv, stream=stream, voronoi_rebuild=rebuild) as sim:
            out[name] = dict(_rate(stream, sim, wv.n, 20, 50),
                             config={"workload": wv.name, "rule": "voronoi", "eta": 0.1,
                                     "voronoi_rebuild": rebuild})
    wp = W.precision_study("voronoi")
    with vk.from_workload(wp, stream=stream) as sim:
        out["voronoi_uniform1M_rho2"] = dict(_rate(stream, sim, wp.n, 5, 10),
                                             config={"workload": wp.name, "rule": "voronoi", "eta": wp.eta})
    wc = W.clustered_large()
    with vk.from_workload(wc, stream=stream, rule="metric", r0=1.0, cell_occupancy=256.0) as sim:
        out["metric_clustered4M_r1"] = dict(_rate(stream, sim, wc.n, 5, 20),
                                            config={"workload": wc.name, "rule": "metric", "r0": 1.0})
    with vk.from_workload(wc, stream=stream, fov=1, fov_cos=0.0, cell_occupancy=256.0) as sim:
        out["knn_fov_clustered4M_halfplane"] = dict(_rate(stream, sim, wc.n, 5, 20),
                                                    config={"workload": wc.name, "rule": "knn", "k": 7,
                                                            "fov_cos": 0.0})
    w3 = W.knn_3d()
    with vk.from_workload(w3, stream=stream) as sim:
        out["knn3d_1M"] = dict(_rate(stream, sim, w3.n, 5, 20), config={"workload": w3.name, "rule": "knn",
                                                                        "k": 7, "dim": 3})
    wv3 = W.voronoi_3d()
    with vk.from_workload(wv3, stream=stream) as sim:
        out["voronoi3d_256k"] = dict(_rate(stream, sim, wv3.n, 3, 10),
                                     config={"workload": wv3.name, "rule": "voronoi", "dim": 3, "eta": wv3.eta})
    # the tissue model's energy and forces of a uniform state: wall time of the
    # whole synchronous call (scratch allocation, three kernels, copies to host)
    wt = W.uniform_system(1 << 20, 1024.0, 16, 2, input_seed=1011, rule="voronoi", k=0)
    with vk.from_workload(wt, stream=stream) as sim:
        sim.tissue(1.0, 1.0, 1.0, 3.8)  # warm-up
        t0 = time.perf_counter()
        for _ in range(3):
            sim.tissue(1.0, 1.0, 1.0, 3.8)
        sec = (time.perf_counter() - t0) / 3
        out["tissue_forces_uniform1M"] = {"value": wt.n / sec, "unit": "particles/s (areas, perimeters, energy, "
                                          "forces per call)", "ms_per_call": sec * 1e3,
                                          "config": {"workload": wt.name, "KA": 1.0, "KP": 1.0, "A0": 1.0,
                                                     "P0": 3.8}}
    return out


# ---------------------------------------------------------------------------
# secondary scenarios (not the benchmark line): batched replicas against
# per-replica launches, the Voronoi rule, the 3D kNN rule
# ---------------------------------------------------------------------------
def _timed(stream, fn):
    import torch
    a = torch.cuda.Event(enable_timing=True)
    b = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    a.record(stream)
    fn()
    b.record(stream)
    b.synchronize()
    return a.elapsed_time(b)


def run_scenario(args):
    import torch
    from paper_2103_10239_gb300 import vk, _build
    from paper_2103_10239_gb300 import workloads as W
    _build.build()
    torch.cuda.set_device(0)
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    out = {"scenario": args.scenario, "steps": args.steps, "warmup": args.warmup, "data": "synthetic"}
    if args.scenario == "replicas":
        ws = W.replica_batch()
        total = sum(w.n for w in ws)
        sim = vk.batch_from_workloads(ws, stream=stream)
        sim.set_graph_steps(args.steps)
        sim.step(args.steps)  # warm-up (and graph capture)
        ms_b = _timed(stream, lambda: sim.step(args.steps)) / args.steps
        sim.close()
        sims = [vk.from_workload(w, stream=stream) for w in ws]
        for x in sims:
            x.step(args.warmup)

        def per_rep():
            for _ in range(args.steps):
                for x in sims:
                    x.step(1)
        ms_p = _timed(stream, per_rep) / args.steps
        for x in sims:
            x.set_graph_steps(args.steps)
            x.step(args.steps)  # capture
        ms_g = _timed(stream, lambda: [x.step(args.steps) for x in sims]) / args.steps
        for x in sims:
            x.close()
        out.update({"metric": "particle-steps/s, 512 replicas (batched launch + multi-step graph)",
                    "value": total / (ms_b * 1e-3), "unit": "particle-steps/s", "ms_per_step": ms_b,
                    "per_replica_launches": {"value": total / (ms_p * 1e-3), "ms_per_step": ms_p},
                    "per_replica_graphs": {"value": total / (ms_g * 1e-3), "ms_per_step": ms_g},
                    "speedup_vs_per_replica_launches": ms_p / ms_b,
                    "speedup_vs_per_replica_graphs": ms_g / ms_b,
                    "config": {"workload": "512 replicas, N_r log-uniform [1024, 65536], k=7, F=16",
                               "n_total": total}})
    else:
        kw = {"n": args.scenario_n} if args.scenario_n > 0 else {}
        if args.scenario == "voronoi":
            w = W.voronoi_mixed(eta=0.1)
        elif args.scenario == "voronoi3d":
            w = W.voronoi_3d(**kw)
        else:
            w = W.knn_3d(**kw)
        over = {} if args.voronoi3_kernel is None else {"voronoi3_kernel": args.voronoi3_kernel}
        sim = vk.from_workload(w, stream=stream, **over)
        sim.step(args.warmup)
        ms = _timed(stream, lambda: sim.step(args.steps)) / args.steps
        sim.set_profiling(True)
        sim.step(3)
        prof = sim.profile()
        sim.close()
        out.update({"metric": f"particle-steps/s ({w.rule}, {w.dim}D)", "value": w.n / (ms * 1e-3),
                    "unit": "particle-steps/s", "ms_per_step": ms,
                    "config": dict({"workload": w.name, "n": w.n, "rule": w.rule, "k": w.k, "dim": w.dim}, **over),
                    "phases_ms_per_step": {k: v[0] / 3 for k, v in prof.items() if v[1]}})
        if not args.no_cpu_baseline:
            out["cpu_baseline"] = scenario_cpu_baseline(w, args.cpu_seconds)
    print(json.dumps(out), flush=True)


def main():
    args = parse()
    if args.scenario != "headline":
        run_scenario(args)
        return
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    dist = None
    if world > 1:
        import torch.distributed as td
        td.init_process_group("nccl")
        dist = td
    run_ours(args, rank, world, dist)
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
