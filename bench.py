#!/usr/bin/env python3
"""Benchmark: exact typed 3+4-node graphlet counting, edges per second.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                    [--workload cl_large|sbm_typed|er_small]

One step = the whole counting path on one graph resident in HBM: tg_build
(device preprocessing) + tg_count(k=4) (per-edge uint32 rows and global
int64 totals, both written to HBM) + tg_free.  value = edges of all ranks /
max-over-ranks time of K steps (CUDA events on the launching stream, barrier
and synchronize on both sides).  The inputs and outputs (CSR 176 MB, per-edge
rows 12.8 GB for the Chung-Lu workload) exceed the 129 MB L2, so no flush is
needed between steps.

e2e: the same metric through the public API with host buffers (pinned CSR
in, per-edge rows and totals out), copies inside the timed region.
cpu_baseline: the CPU oracle (Alg. 1-3 + Lemmas) on the host cores, its
full-graph time extrapolated from a seeded stratified edge sample (every
sampled edge timed), on all cores and on one thread.  --impl reference
times that oracle, with the same estimator, as the reference arm.

Multi-GPU (torchrun): every rank counts its own copy of the workload (edges
are independent problems; weak scaling), no collective on the data path.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "typed-graphlet edges/sec (3+4-node, exact)"
UNIT = "edges/s"
WORKLOADS = {
    "cl_large": "Chung-Lu n=2,000,000 m=20,000,000 gamma=2.1 max weight 5e4, L=5 Zipf(1.2) types",
    "sbm_typed": "SBM 500k/300k/150k/50k nodes, L=4 types, m=30,000,000, affinity 1 between / 0.05 within",
    "er_small": "Erdos-Renyi n=2,000 m=10,000, L=3 uniform types",
    "cl_mid": "Chung-Lu n=200,000 m=2,000,000 gamma=2.1 max weight 1.2e4, L=5 Zipf(1.2) types (profiling size)",
}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="cl_large", choices=sorted(WORKLOADS))
    ap.add_argument("--e2e-steps", type=int, default=2)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--mode", default="plain", choices=["plain", "batched", "serve"],
                    help="plain: one graph (the headline line); batched: the ego-network batch vs per-graph launches")
    ap.add_argument("--graphs", type=int, default=8192, help="graphs in the batched workload")
    ap.add_argument("--tune-graphs", type=int, default=256,
                    help="batched: graphs of the sub-batch the autotuner measures (0: library defaults)")
    ap.add_argument("--rate", type=float, default=200_000 / 60, help="serving: Poisson arrivals per second")
    ap.add_argument("--duration", type=float, default=60.0, help="serving: seconds of measured arrivals")
    ap.add_argument("--serve-warmup", type=float, default=10.0,
                    help="serving: seconds of arrivals before the measured window")
    ap.add_argument("--plain-seconds", type=float, default=10.0,
                    help="serving: measured seconds of the trace replayed by the plain sequential server")
    ap.add_argument("--pool", type=int, default=1024, help="serving: distinct request graphs")
    ap.add_argument("--oracle-fraction", type=float, default=0.02,
                    help="batched / serve: fraction of graphs (requests) whose totals the CPU oracle checks")
    ap.add_argument("--oracle-seconds", type=float, default=240.0,
                    help="batched / serve: oracle time budget of that check (0: no limit)")
    ap.add_argument("--position-aware", action="store_true",
                    help="plain mode: also time the position-aware count (Sec. 5) of the same graph")
    ap.add_argument("--edge-typed", action="store_true",
                    help="plain mode: also time the edge-typed 3-node count of the workload, 4 seeded edge types")
    ap.add_argument("--directed", action="store_true",
                    help="plain mode: also time the directed typed 3-node count (Sec. 4.8) of the workload's "
                         "edges oriented by a seeded coin")
    return ap.parse_args()


# ----------------------------------------------------------------- helpers

class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.samples = []
        self._stop = threading.Event()
        self._proc = None
        self._thread = None

    def start(self):
        try:
            self._proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except (OSError, FileNotFoundError):
            self._proc = None
            return
        self._thread = threading.Thread(target=self._read, daemon=True)
        self._thread.start()

    def _read(self):
        for line in self._proc.stdout:
            self.samples.append([x.strip() for x in line.split(",")])
            if self._stop.is_set():
                break

    def stop(self) -> dict:
        self._stop.set()
        if self._proc:
            self._proc.terminate()
            try:
                self._proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self._proc.kill()
        if not self.samples:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        sm = [float(s[1]) for s in self.samples if s[1].replace(".", "", 1).isdigit()]
        smax = [float(s[2]) for s in self.samples if s[2].replace(".", "", 1).isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for s in self.samples for k in range(4) if len(s) > 5 + k and s[5 + k] == "Active"})
        power = [float(s[3]) for s in self.samples if s[3].replace(".", "", 1).isdigit()]
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": reasons, "samples": len(self.samples),
                "power_w_max": max(power) if power else None}


def gpu_local_cpus(index: int) -> list | None:
    """Host CPUs attached to GPU `index` (its PCI device's local_cpulist),
    or None when that cannot be read."""
    try:
        bus = subprocess.run(["nvidia-smi", "-i", str(index), "--query-gpu=pci.bus_id", "--format=csv,noheader"],
                             capture_output=True, text=True, timeout=30).stdout.strip()
        dom, rest = bus.split(":", 1)
        path = f"/sys/bus/pci/devices/{dom[-4:].lower()}:{rest.lower()}/local_cpulist"
        with open(path) as f:
            spec = f.read().strip()
        cpus = []
        for part in spec.split(","):
            a, _, b = part.partition("-")
            cpus += list(range(int(a), int(b or a) + 1))
        allowed = os.sched_getaffinity(0)
        cpus = [c for c in cpus if c in allowed]
        return cpus or None
    except (OSError, ValueError, subprocess.SubprocessError):
        return None


class NearGpu:
    """Runs a block on the host CPUs attached to the GPU, so that pinned
    buffers allocated inside it are placed in that CPU's memory (first touch)
    and host-device copies take the direct link; restores the affinity."""

    def __init__(self, index: int):
        self.cpus = gpu_local_cpus(index)
        self.saved = None

    def __enter__(self):
        if self.cpus:
            self.saved = os.sched_getaffinity(0)
            os.sched_setaffinity(0, self.cpus)
        return self

    def __exit__(self, *exc):
        if self.saved is not None:
            os.sched_setaffinity(0, self.saved)
        return False


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


# DRAM bytes (read + write) per launch of a kernel, from the ncu capture
# summarised under profiles/ for that workload and the current kernel code
# (an entry is removed when its kernel changes).
TRAFFIC = {("cl_large", "k_wedge_hub"): 230.590e9, ("cl_large", "k_sum"): 52.625e9, ("cl_large", "k_epi4"): 36.473e9}


def w_alg_bytes(g: dict, tsize, S: int) -> dict:
    """The algorithmic traffic model W_alg = sum_e [4(d_i + d_j) +
    sum_{w in U_e} 4 min(d_w, |U_e| ceil(log2 d_w))] + 4 S m: per edge both
    rows, then for every node of U_e = (Gamma_i u Gamma_j) minus {i, j} the cheaper
    of scanning its row or searching U_e's members in it, plus the rows
    written.  |U_e| = d_i + d_j - 2 - |T_e| (|T_e| from the counts); the sum
    over U_e is taken over Gamma_i minus {j} and Gamma_j minus {i}, so the
    nodes of T_e count twice: an upper bound."""
    rp, col, n = g["row_ptr"], g["col"].astype(np.int64), g["n"]
    deg = np.diff(rp).astype(np.int64)
    lg = np.zeros(n, np.int64)
    lg[deg > 1] = np.ceil(np.log2(deg[deg > 1])).astype(np.int64)
    rows = np.repeat(np.arange(n, dtype=np.int64), deg)
    dw, lw = deg[col], lg[col]
    # threshold of each entry: min(d_w, U lg_w) = d_w exactly when U >= d_w / lg_w
    r = np.where(lw > 0, dw / np.maximum(lw, 1), np.inf)
    order = np.lexsort((r, rows))
    r_s, d_s, l_s = r[order], dw[order].astype(np.float64), lw[order].astype(np.float64)
    cd = np.concatenate([[0.0], np.cumsum(d_s)])
    cl = np.concatenate([[0.0], np.cumsum(l_s)])
    up = col > rows
    src, dst = rows[up], col[up]
    o2 = np.lexsort((dst, src))
    src, dst = src[o2], dst[o2]
    U = (deg[src] + deg[dst] - 2 - np.asarray(tsize, dtype=np.int64)).astype(np.float64)
    key = np.where(np.isinf(r_s), 4e15, rows[order] * 1e9 + np.minimum(r_s, 5e8))

    def side(x, other):
        lo = rp[x].astype(np.int64)
        hi = rp[x + 1].astype(np.int64)
        k = np.searchsorted(key, x * 1e9 + U, side="right")
        k = np.clip(k, lo, hi)
        tot = (cd[k] - cd[lo]) + U * (cl[hi] - cl[k])
        # drop the other endpoint, which is in Gamma_x but not in U_e
        dd, ll = deg[other].astype(np.float64), lg[other].astype(np.float64)
        return tot - np.minimum(dd, U * ll)

    s = 4.0 * (deg[src] + deg[dst]).sum() + 4.0 * (side(src, dst).sum() + side(dst, src).sum())
    return {"bytes": float(s + 4.0 * S * len(src)), "model": "upper bound (nodes of T counted from both sides)"}


def kernel_units(g: dict, light_anchor_max: int = 64, hub_min: int = 1 << 14) -> dict:
    """Work units of the count kernels, computed on the host from the graph:
    degree-priority wedges (the search for the 4-cycles behind P) split
    by the anchor class the build assigns (light: at most light_anchor_max
    wedges; hub: more than hub_min; the defaults are the library's
    tg_options light_anchor_max_wedges and hub_min_wedges), oriented
    (anchor, neighbour) pairs per class, and the shorter side of every
    typed intersection, sum_e sum_t min(d_i^t, d_j^t)."""
    rp, col, ty, n, L = g["row_ptr"], g["col"].astype(np.int64), g["types"], g["n"], g["L"]
    deg = np.diff(rp)
    rank = np.empty(n, np.int64)
    rank[np.lexsort((np.arange(n), deg))] = np.arange(n)     # priority = (degree, id)
    rows = np.repeat(np.arange(n, dtype=np.int64), deg)
    key = np.sort(rows * n + rank[col])                       # each row by neighbour priority
    up = rank[col] < rank[rows]                               # (anchor x, lower-priority neighbour v)
    x, v = rows[up], col[up]
    cnt = np.searchsorted(key, v * n + rank[x]) - rp[v]       # wedges x - v - w with w below x
    W = np.bincount(x, weights=cnt, minlength=n)
    light = (W > 0) & (W <= light_anchor_max)
    heavy = (W > light_anchor_max) & (W <= hub_min)
    hub = W > hub_min
    pairs = np.bincount(x, minlength=n)
    tdeg = np.zeros((n, L), np.int64)
    np.add.at(tdeg, (rows, ty[col].astype(np.int64)), 1)
    lo = col > rows
    mins = np.minimum(tdeg[rows[lo]], tdeg[col[lo]]).sum()
    return {"wedges_light": float(W[light].sum()), "wedges_heavy": float(W[heavy].sum()),
            "wedges_hub": float(W[hub].sum()), "pairs_light": float(pairs[light].sum()),
            "pairs_heavy": float(pairs[heavy].sum()), "pairs_hub": float(pairs[hub].sum()), "hubs": int(hub.sum()),
            "typed_min_sum": float(mins)}


def clique_units(pe, L: int, big_t: int = 256, chunk: int = 1 << 22) -> dict:
    """|T_e| (sum of the triangle slots) and K_e (sum of the 4-clique orbit
    slots g12) of every edge, read from the per-edge rows, summed over the
    edges of at most and of more than big_t triangles."""
    import torch
    P = L * (L + 1) // 2
    k0 = 2 * L + 9 * P
    out = {"t_small": 0, "t_big": 0, "k_small": 0, "k_big": 0, "edges_big": 0}
    for a in range(0, pe.shape[0], chunk):
        rows = pe[a:a + chunk]
        T = rows[:, L:2 * L].long().sum(1)
        K = rows[:, k0:k0 + P].long().sum(1)
        big = T > big_t
        out["t_small"] += int(T[~big].sum())
        out["t_big"] += int(T[big].sum())
        out["k_small"] += int(K[~big].sum())
        out["k_big"] += int(K[big].sum())
        out["edges_big"] += int(big.sum())
    return out


def algorithmic_bytes(u: dict, n: int, m: int, L: int, S: int, tri_rows: int) -> dict:
    """Bytes each count kernel must move at least once in this formulation
    (every element of its inputs read once, however often L2 serves it again,
    and every element of its outputs written once), per launch over the whole
    graph; tri_rows: (edge, type) pairs with a triangle, whose rows of sums are
    kept.
      k_tri       per edge: its entry of the N+ lists read 8 (id, edge id);
                  its row of typed triangle counts zeroed and written 64;
      k_sum_zero  per edge its row of triangle counts read 32, per kept row
                  16L written;
      k_sum       per edge its entry of the N+ lists 8 and row of triangle
                  counts 32, per node its typed degrees 32, per kept row its
                  sums read and written 32L;
      k_slot_rows per adjacency slot L^2 values read and written 8L^2;
      k_epi4      per edge: endpoints and slots 24, its row of triangle counts
                  32, two rows of 4-cycle values 8L^2, its output row 4S; per
                  node its type offsets 4(L+1), delta and tau 8L^2 (32-bit);
                  per kept row its sums 16L.
    Of the wedge kernels, whose updates scatter over more than L2 holds, the
    accesses instead:
      k_wedge_light, k_wedge_64 to k_wedge_1024 (one line, k_wedge_shared):
                  per wedge the far node's id 4 + its 4-cycle slot 4 read +
                  4 written; per (anchor, neighbour) pair: L slots 8 B each;
      k_wedge_hub when the library's work counters give them: per hub wedge
                  its far node's id 4, per nonzero 4-cycle slot update (a
                  wedge and a type of the fourth node, or a (hub, neighbour,
                  type) sum) the slot read and written 8."""
    LL = L * L
    return {
        "k_tri": 72.0 * m,
        "k_sum_zero": 32.0 * m + 16.0 * L * tri_rows,
        "k_sum": 40.0 * m + 32.0 * n + 32.0 * L * tri_rows,
        "k_wedge_shared": 12.0 * (u["wedges_light"] + u["wedges_heavy"]) + 8.0 * L * (u["pairs_light"] + u["pairs_heavy"]),
        "k_wedge_hub": 4.0 * u["hub_wedges_counted"] + 8.0 * u["hub_slot_updates"] if "hub_slot_updates" in u else
        12.0 * u["wedges_hub"] + 8.0 * L * u["pairs_hub"],
        "k_slot_rows": 16.0 * LL * m,
        "k_epi4": (24.0 + 32 + 8 * LL + 4 * S) * m + (4.0 * (L + 1) + 8 * LL) * n + 16.0 * L * tri_rows,
    }


def count_only(m: int, count_ms: float, step_ms: float) -> dict | None:
    """Edges per second of tg_count alone (CUDA events around the call, per
    step) and the rest of the step (tg_build, tg_free) in milliseconds."""
    if count_ms <= 0:
        return None
    return {"value": round(m / (count_ms / 1e3), 1), "unit": UNIT, "count_ms": round(count_ms, 3),
            "build_and_free_ms": round(max(step_ms - count_ms, 0.0), 3)}


# ------------------------------------------------------------- our arm

def run_ours(args):
    import torch

    import graphgen
    import paper_2010_14058_gb300 as tg

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    dist = None
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    dev = torch.device("cuda", torch.cuda.current_device())

    from paper_2010_14058_gb300 import build as tgbuild
    tgbuild.build()
    g = graphgen.workload(args.workload)
    L, m = g["L"], g["m"]
    lay = tg.tg_layout(L, 4)
    S, G = lay["per_edge_slots"], lay["global_slots"]
    units = kernel_units(g) if rank == 0 else None
    rp, col, ty = tg.to_device(g, dev)
    pe = torch.empty((m, S), dtype=torch.int32, device=dev)
    gl = torch.empty(G, dtype=torch.int64, device=dev)
    stream = torch.cuda.current_stream(dev)

    def barrier():
        if dist is not None:
            dist.barrier()

    kernel_ms, count_ms_sum = {}, [0.0]
    ksteps = min(args.steps, 5)
    launches = [0]

    def one(build, count, kernels=None, events=None):
        """build, count, status, free; `kernels`: with the library's per-kernel timing, which runs the kernels one
        after another; `events`: recorded around the count."""
        h = build()
        launches[0] += h.last_launch_count
        if kernels is not None:
            tg.tg_set_timing(h, True)
        if events:
            events[0].record(stream)
        count(h)
        if events:
            events[1].record(stream)
        launches[0] += h.last_launch_count
        if kernels is not None:
            for name, (ms, n) in tg.tg_get_timing(h).items():
                a = kernels.setdefault(name, [0.0, 0])
                a[0] += ms
                a[1] += n
        st = tg.tg_query_status(h)
        if events:
            count_ms_sum[0] += events[0].elapsed_time(events[1])
        h.free()
        return st

    def timed_steps(build, count, kernels):
        """Milliseconds of args.steps steps after the warm-up, and their status; then, untimed, the kernels' times."""
        for _ in range(args.warmup):
            one(build, count)
        torch.cuda.synchronize()
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        st = 0
        for _ in range(args.steps):
            st = one(build, count) or st
        b.record(stream)
        torch.cuda.synchronize()
        for _ in range(ksteps):
            st = one(build, count, kernels=kernels) or st
        return a.elapsed_time(b), st

    def step(kernels=None, events=None):
        return one(lambda: tg.tg_build(rp, col, ty, L, stream=stream),
                   lambda h: tg.tg_count(h, 4, pe, gl, stream=stream), kernels, events)

    for _ in range(args.warmup):
        step()
    status = 0
    count_ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    # timed region
    clocks = ClockSampler(torch.cuda.current_device())
    barrier()
    torch.cuda.synchronize()
    clocks.start()
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    launches[0] = 0
    t0.record(stream)
    for _ in range(args.steps):
        st = step(events=count_ev)
        status = status or st
    t1.record(stream)
    torch.cuda.synchronize()
    barrier()
    n_launches = launches[0]
    clk = clocks.stop()
    ms = t0.elapsed_time(t1)
    ms_t = torch.tensor([ms], dtype=torch.float64, device=dev)
    if dist is not None:
        dist.all_reduce(ms_t, op=dist.ReduceOp.MAX)
    ms_max = float(ms_t.item())
    value = world * m * args.steps / (ms_max / 1e3)

    # end-to-end figures first, right after the timed region (before the
    # roofline work below allocates anything)
    # end to end through host buffers (pinned buffers in the memory of the
    # host CPUs attached to this GPU)
    e2e = None
    near = NearGpu(torch.cuda.current_device())
    near.__enter__()
    if not args.no_e2e and rank == 0:
        h_rp = torch.from_numpy(np.ascontiguousarray(g["row_ptr"])).pin_memory()
        h_col = torch.from_numpy(np.ascontiguousarray(g["col"])).pin_memory()
        h_ty = torch.from_numpy(np.ascontiguousarray(g["types"])).pin_memory()
        h_pe = torch.empty((m, S), dtype=torch.int32).pin_memory()
        h_gl = torch.empty(G, dtype=torch.int64).pin_memory()

        def e2e_step():
            h = tg.tg_build(h_rp, h_col, h_ty, L, stream=stream)
            tg.tg_count(h, 4, h_pe, h_gl, stream=stream)
            h.free()

        for _ in range(max(1, min(args.warmup, 2))):     # untimed: staging buffers, first touch of pinned pages
            e2e_step()
        torch.cuda.synchronize()
        step_ms = []
        t = time.perf_counter()
        for _ in range(args.e2e_steps):
            t_s = time.perf_counter()
            e2e_step()                                   # returns after its rows are in host memory
            step_ms.append(round(1e3 * (time.perf_counter() - t_s), 1))
        torch.cuda.synchronize()
        el = time.perf_counter() - t
        bi = h_rp.numel() * 8 + h_col.numel() * 4 + h_ty.numel()
        bo = h_pe.numel() * 4 + h_gl.numel() * 8
        e2e = {"value": round(m * args.e2e_steps / el, 1), "unit": UNIT, "h2d_bytes_per_step": int(bi),
               "d2h_bytes_per_step": int(bo), "step_ms": step_ms}

    # the same end to end with the sparse per-edge form (only nonzero counts
    # cross PCIe: row offsets, uint16 slots, uint32 counts)
    e2e_sparse = None
    if not args.no_e2e and rank == 0:
        h = tg.tg_build(h_rp, h_col, h_ty, L, stream=stream)
        d_off = torch.empty(m + 1, dtype=torch.int64, device=dev)
        nnz = tg.tg_count_sparse(h, 4, d_off, stream=stream)
        h.free()
        d_slot = torch.empty(nnz, dtype=torch.int16, device=dev)
        d_val = torch.empty(nnz, dtype=torch.int32, device=dev)
        d_gl = torch.empty(G, dtype=torch.int64, device=dev)
        p_off = torch.empty(m + 1, dtype=torch.int64).pin_memory()
        p_slot = torch.empty(nnz, dtype=torch.int16).pin_memory()
        p_val = torch.empty(nnz, dtype=torch.int32).pin_memory()

        def e2e_sparse_step():
            h = tg.tg_build(h_rp, h_col, h_ty, L, stream=stream)
            tg.tg_count_sparse(h, 4, d_off, d_slot, d_val, d_gl, stream=stream)
            with torch.cuda.stream(stream):
                p_off.copy_(d_off, non_blocking=True)
                p_slot.copy_(d_slot, non_blocking=True)
                p_val.copy_(d_val, non_blocking=True)
                h_gl.copy_(d_gl, non_blocking=True)
            h.free()

        for _ in range(max(1, min(args.warmup, 2))):
            e2e_sparse_step()
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(args.e2e_steps):
            e2e_sparse_step()
        torch.cuda.synchronize()
        el = time.perf_counter() - t
        bo = p_off.numel() * 8 + nnz * 6 + G * 8
        e2e_sparse = {"value": round(m * args.e2e_steps / el, 1), "unit": UNIT, "h2d_bytes_per_step": int(bi),
                      "d2h_bytes_per_step": int(bo), "nonzero_pairs": int(nnz),
                      "pairs_per_edge": round(nnz / max(m, 1), 2)}
    near.__exit__(None, None, None)
    if e2e is not None:
        e2e["host_cpus"] = (f"{len(near.cpus)} CPUs attached to the GPU ({near.cpus[0]}-{near.cpus[-1]})"
                            if near.cpus else "unpinned (no local CPU list)")


    # roofline: algorithmic bytes of each count kernel per step over its
    # CUDA-event time per step (untimed steps of their own: per-kernel timing
    # runs the kernels one after another)
    peak, peak_kind = load_peaks()
    roofline, per_kernel, compulsory, count_alone, walg, work = None, {}, None, None, None, None
    if rank == 0:
        for _ in range(ksteps):
            status = step(kernels=kernel_ms) or status
        # the hub wedges and 4-clique words of one count, from the library's work counters
        # (one extra, untimed count)
        h = tg.tg_build(rp, col, ty, L, stream=stream)
        tg.tg_set_work_counting(h, True)
        tg.tg_count(h, 4, pe, gl, stream=stream)
        work = tg.tg_get_work(h)
        h.free()
        cu = clique_units(pe, L)
        units.update({"clique": cu})
        if work.get("hub_wedges"):
            units.update({"hub_wedges_counted": float(work["hub_wedges"]),
                          "hub_slot_updates": float(work["hub_slot_updates"])})
        tri_rows = sum(int((pe[a:a + (1 << 22), L:2 * L] != 0).sum()) for a in range(0, m, 1 << 22))
        abytes = algorithmic_bytes(units, g["n"], m, L, S, tri_rows)
        # the shared-memory wedge forms share one bound
        forms = [v for k, v in kernel_ms.items() if k.startswith("k_wedge_") and k != "k_wedge_hub"]
        timed = {k: v for k, v in kernel_ms.items() if v not in forms}
        if forms:
            timed["k_wedge_shared"] = (sum(v[0] for v in forms), sum(v[1] for v in forms))
        for name, (kms, nl) in timed.items():
            if abytes.get(name) is None or kms <= 0:
                continue
            step_ms = kms / ksteps
            gbs = abytes[name] / (step_ms / 1e3) / 1e9
            per_kernel[name] = {"ms_per_step": round(step_ms, 3), "launches_per_step": nl // ksteps,
                                "algorithmic_gb": round(abytes[name] / 1e9, 3), "achieved_gbs": round(gbs, 2),
                                "frac": round(gbs / peak, 5)}
        top = max(timed.items(), key=lambda kv: kv[1][0])[0]
        if top in per_kernel and "achieved_gbs" in per_kernel[top]:
            pk = per_kernel[top]
            roofline = {"kernel": top, "bound": "hbm", "achieved": pk["achieved_gbs"], "peak": peak,
                        "peak_kind": peak_kind, "unit": "GB/s", "frac": pk["frac"],
                        "algorithmic_bytes": abytes[top], "ms_per_step": pk["ms_per_step"],
                        "traffic": TRAFFIC.get((args.workload, top))}
            if roofline["traffic"]:
                # the measured DRAM bytes of a launch over its CUDA-event time
                roofline["traffic_frac"] = round(roofline["traffic"] / (pk["ms_per_step"] / 1e3) / 1e9 / peak, 5)
        # compulsory traffic of the whole count: CSR and types read once,
        # outputs written once -- the headline "% of HBM roofline"
        cb = 8.0 * m + 8.0 * g["n"] + g["n"] + 4.0 * S * m + 8.0 * G
        count_ms = count_ms_sum[0] / args.steps
        compulsory = {"bound": "hbm", "bytes": cb, "count_ms": round(count_ms, 3), "peak": peak,
                      "peak_kind": peak_kind, "unit": "GB/s",
                      "achieved": round(cb / (count_ms / 1e3) / 1e9, 2),
                      "frac": round(cb / (count_ms / 1e3) / 1e9 / peak, 6)}
        count_alone = count_only(m, count_ms, ms_max / args.steps)
        tsize = pe[:, L:2 * L].sum(dim=1, dtype=torch.int64).cpu().numpy()
        walg = w_alg_bytes(g, tsize, S)
        walg["per_s_gb"] = round(walg["bytes"] / (count_ms / 1e3) / 1e9, 2)
        walg["frac_of_hbm_peak"] = round(walg["per_s_gb"] / peak, 4)
        walg["note"] = "effective algorithmic bandwidth W_alg / T_count; may exceed HBM (L2 and shared-memory reuse)"
    kernel_share = {k: round(v[0] / sum(x[0] for x in kernel_ms.values()), 4) for k, v in kernel_ms.items()}

    # position-aware counts (Sec. 5) of the same graph: same gathering
    # passes, position-aware epilogue, rows of S_pa slots
    position_aware = None
    if args.position_aware and rank == 0:
        lay_pa = tg.tg_pa_layout(L)
        pe_pa = torch.empty((m, lay_pa["per_edge_slots"]), dtype=torch.int32, device=dev)
        gl_pa = torch.empty(lay_pa["global_slots"], dtype=torch.int64, device=dev)
        pa_ms = {}
        pms, pa_status = timed_steps(lambda: tg.tg_build(rp, col, ty, L, stream=stream),
                                     lambda h: tg.tg_count_position_aware(h, pe_pa, gl_pa, stream=stream), pa_ms)
        position_aware = {"value": round(m * args.steps / (pms / 1e3), 1), "unit": UNIT,
                          "ms_per_step": round(pms / args.steps, 3), "status": tg.STATUS[pa_status],
                          "per_edge_slots": lay_pa["per_edge_slots"], "global_slots": lay_pa["global_slots"],
                          "k_epi4_pa_ms_per_step": round(pa_ms.get("k_epi4_pa", [0.0])[0] / ksteps, 3),
                          "k_epi4_ms_per_step": round(kernel_ms.get("k_epi4", [0.0])[0] / ksteps, 3),
                          "step": "tg_build + tg_count_position_aware + tg_free, device-resident"}

    # directed typed 3-node counts (Sec. 4.8) of the same edges, each oriented
    # by a seeded coin: tg_build_directed + tg_count_directed3 per step
    directed = None
    if args.directed and rank == 0:
        src_e, dst_e = edge_list(g)
        flip = np.random.default_rng(CPU_SEED + 48).random(len(src_e)) < 0.5
        tail = np.where(flip, dst_e, src_e)
        head = np.where(flip, src_e, dst_e)
        order = np.argsort(tail, kind="stable")
        d_rp = torch.as_tensor(np.concatenate([[0], np.cumsum(np.bincount(tail, minlength=g["n"]))]).astype(np.int64),
                               device=dev)
        d_col = torch.as_tensor(head[order].astype(np.int32), device=dev)
        lay_d = tg.tg_directed_layout(L)
        pe_d = torch.empty((m, lay_d["per_edge_slots"]), dtype=torch.int32, device=dev)
        gl_d = torch.empty(lay_d["global_slots"], dtype=torch.int64, device=dev)
        d_ms = {}
        dms, d_status = timed_steps(lambda: tg.tg_build_directed(d_rp, d_col, ty, L, stream=stream),
                                    lambda h: tg.tg_count_directed3(h, pe_d, gl_d, stream=stream), d_ms)
        directed = {"value": round(m * args.steps / (dms / 1e3), 1), "unit": UNIT,
                    "ms_per_step": round(dms / args.steps, 3), "status": tg.STATUS[d_status],
                    "per_edge_slots": lay_d["per_edge_slots"], "global_slots": lay_d["global_slots"],
                    "kernels_ms_per_step": {k: round(v[0] / ksteps, 3) for k, v in d_ms.items()},
                    "step": "tg_build_directed + tg_count_directed3 + tg_free, device-resident; each edge of the "
                            "workload oriented by a seeded coin"}

    # edge-typed 3-node counts (Def. 1's edge types) of the same graph, 4
    # seeded edge types: tg_build_edge_typed + tg_count_edge_typed3 per step
    edge_typed = None
    if args.edge_typed and rank == 0:
        X = 4
        xi = torch.as_tensor(graphgen.edge_types(g, X, CPU_SEED + 49), device=dev)
        lay_x = tg.tg_edge_typed_layout(L, X)
        pe_x = torch.empty((m, lay_x["per_edge_slots"]), dtype=torch.int32, device=dev)
        gl_x = torch.empty(lay_x["global_slots"], dtype=torch.int64, device=dev)
        x_ms = {}
        xms, x_status = timed_steps(lambda: tg.tg_build_edge_typed(rp, col, ty, xi, L, X, stream=stream),
                                    lambda h: tg.tg_count_edge_typed3(h, pe_x, gl_x, stream=stream), x_ms)
        edge_typed = {"value": round(m * args.steps / (xms / 1e3), 1), "unit": UNIT,
                      "ms_per_step": round(xms / args.steps, 3), "status": tg.STATUS[x_status], "edge_types": X,
                      "per_edge_slots": lay_x["per_edge_slots"], "global_slots": lay_x["global_slots"],
                      "kernels_ms_per_step": {k: round(v[0] / ksteps, 3) for k, v in x_ms.items()},
                      "step": "tg_build_edge_typed + tg_count_edge_typed3 + tg_free, device-resident; each edge "
                              "of the workload typed by a seeded hash"}

    cpu = None
    if not args.no_cpu and rank == 0 and world == 1:
        cpu = cpu_baseline(g)

    if rank == 0:
        line = {
            "metric": METRIC, "value": round(value, 1), "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": round(ms_max / args.steps, 3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "int64", "data": "synthetic",
            "config": {"workload": args.workload, "description": WORKLOADS[args.workload], "nodes": g["n"],
                       "edges": m, "types": L, "k": 4, "per_edge_slots": S, "global_slots": G,
                       "l2": "inputs and outputs larger than L2 (no flush)",
                       "step": "tg_build + tg_count(k=4) + tg_free, device-resident inputs and outputs"},
            "status": tg.STATUS[status], "roofline": roofline, "hbm_roofline": compulsory,
            "kernel_roofline": per_kernel, "w_alg": walg, "work": work,
            "count_only": count_alone, "kernel_share": kernel_share,
            "units": units,
            "cpu_baseline": cpu, "e2e": e2e, "e2e_sparse": e2e_sparse, "clocks": clk,
            "gpu_launches": int(n_launches),
        }
        if position_aware is not None:
            line["position_aware"] = position_aware
        if directed is not None:
            line["directed"] = directed
        if edge_typed is not None:
            line["edge_typed"] = edge_typed
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


# --------------------------------------------------------- CPU oracle arm
#
# The oracle cannot count the benchmark graph in full within a benchmark run
# (about 16 days on one core), so both arms estimate its full-graph time
# from a seeded stratified sample of edges:
#   * work proxy of edge (u, v): d_u + d_v + s_u + s_v, s_x = sum of the
#     degrees of x's neighbours -- the oracle marks both neighbourhoods and
#     scans every neighbour's row (Alg. 1-3), so its time per edge follows
#     this proxy closely;
#   * a certainty stratum of the `heaviest` edges by proxy, timed in full;
#     the other edges in strata by floor(log2(proxy)), each sampled without
#     replacement, n_h proportional to the stratum's share of the proxy
#     total (at least 3);
#   * every sampled edge timed by the thread that counts it; the full-graph
#     time T = T_open + sum_h (N_h / n_h) * (sum of the stratum's sampled
#     times) / C, C = threads (a Horvitz-Thompson estimate; with C threads
#     the per-edge times are taken under C-thread load, and the full graph's
#     20M edges balance across the threads, so no idle time is added);
#   * T_open = the one-off graph preparation (copy, row sort, validation).
# The single-thread figure uses a subsample (every `thin`-th edge of each
# stratum sample) to stay within the time budget.

CPU_SEED = 20201029


def edge_list(g: dict):
    """(src, dst) of every edge in edge-id order (u < v, lexicographic)."""
    rp, col, n = g["row_ptr"], g["col"].astype(np.int64), g["n"]
    rows = np.repeat(np.arange(n, dtype=np.int64), np.diff(rp))
    up = col > rows
    src, dst = rows[up], col[up]
    order = np.lexsort((dst, src))
    return src[order], dst[order]


def edge_cost_proxy(g: dict):
    """(src, dst, proxy) of every edge in edge-id order (u < v, lexicographic)."""
    rp, col, n = g["row_ptr"], g["col"].astype(np.int64), g["n"]
    deg = np.diff(rp)
    rows = np.repeat(np.arange(n, dtype=np.int64), deg)
    s = np.bincount(rows, weights=deg[col], minlength=n)
    up = col > rows
    src, dst = rows[up], col[up]
    order = np.lexsort((dst, src))
    src, dst = src[order], dst[order]
    return src, dst, (deg[src] + deg[dst]).astype(np.float64) + s[src] + s[dst]


def oracle_design(proxy, budget_edges: int = 1000, heaviest: int = 100, seed: int = CPU_SEED) -> list:
    """Strata of the estimator: [(name, N_h, sampled edge ids)], seeded."""
    rng = np.random.default_rng(seed)
    m = len(proxy)
    order = np.argsort(-proxy, kind="stable")
    top = np.sort(order[:min(heaviest, m)])
    strata = [("heaviest", len(top), top)] if len(top) else []
    rest = np.sort(order[len(top):])
    if len(rest) == 0:
        return strata
    bins = np.floor(np.log2(np.maximum(proxy[rest], 1.0))).astype(np.int64)
    total = proxy[rest].sum()
    for b in np.unique(bins):
        members = rest[bins == b]
        share = proxy[members].sum() / total if total > 0 else len(members) / len(rest)
        n_h = int(min(len(members), max(3, round(budget_edges * share))))
        pick = np.sort(rng.choice(members, size=n_h, replace=False))
        strata.append((f"log2 proxy {int(b)}", len(members), pick))
    return strata


def oracle_estimate(og, strata, nthreads: int, thin: int = 1, seed: int = CPU_SEED) -> dict:
    """Full-graph oracle time from the sampled edge times (see above)."""
    rng = np.random.default_rng(seed + nthreads)
    ids, w, h_of = [], [], []
    for h, (_, N_h, pick) in enumerate(strata):
        sub = pick[::thin] if thin > 1 else pick
        if thin > 1 and len(sub) < 2:
            sub = pick[:2]
        ids.append(sub)
        w.append(np.full(len(sub), N_h / len(sub)))
        h_of.append(np.full(len(sub), h))
    ids, w, h_of = np.concatenate(ids), np.concatenate(w), np.concatenate(h_of)
    perm = rng.permutation(len(ids))                  # mix heavy and light edges across the threads
    ids, w, h_of = ids[perm], w[perm], h_of[perm]
    t = time.perf_counter()
    _, _, sec = og.paper_edges(ids, k=4, nthreads=nthreads, times=True)
    wall = time.perf_counter() - t
    work = float((w * sec).sum())                     # estimated thread-seconds over all edges
    var = 0.0                                         # stratified variance of that estimate
    for h, (_, N_h, _) in enumerate(strata):
        x = sec[h_of == h]
        if len(x) > 1 and len(x) < N_h:
            var += N_h * N_h * (1 - len(x) / N_h) * x.var(ddof=1) / len(x)
    return {"edges_timed": int(len(ids)), "sample_wall_s": wall, "work_thread_s": work,
            "work_rel_se": float(np.sqrt(var) / work) if work > 0 else 0.0}


def cpu_baseline(g: dict, budget_edges: int = 1000, heaviest: int = 100, thin: int = 10) -> dict:
    """The CPU oracle (Alg. 1-3 + Lemmas, OpenMP over edges, Sec. 4.7)
    timed on the host cores by the stratified estimator: full-graph edges/s
    on all cores (value) and on one thread."""
    import oracle
    m = g["m"]
    _, _, proxy = edge_cost_proxy(g)
    full = m <= 20_000                                  # small graphs: every edge timed, nothing extrapolated
    if full:
        budget_edges, thin = m, 1
    strata = oracle_design(proxy, budget_edges, heaviest)
    t = time.perf_counter()
    og = oracle.OpenGraph(g)
    t_open = time.perf_counter() - t
    cores = oracle.max_threads()
    og.paper_edges(strata[0][2][:min(8, len(strata[0][2]))], nthreads=cores)     # page in the graph
    allc = oracle_estimate(og, strata, cores)
    one = oracle_estimate(og, strata, 1, thin=thin)
    og.close()
    t_all = t_open + allc["work_thread_s"] / cores
    t_one = t_open + one["work_thread_s"]
    n_sample = sum(len(x[2]) for x in strata)
    if full:
        return {"value": round(m / t_all, 2), "unit": UNIT, "cores": cores, "kind": "oracle",
                "value_1thread": round(m / t_one, 2), "full_graph_s": round(t_all, 3),
                "full_graph_s_1thread": round(t_one, 3), "open_s": round(t_open, 3),
                "sample": f"all {m} edges timed (no extrapolation): all cores in {allc['sample_wall_s']:.2f} s, "
                          f"one thread in {one['sample_wall_s']:.2f} s, plus the graph preparation"}
    return {"value": round(m / t_all, 2), "unit": UNIT, "cores": cores, "kind": "oracle",
            "value_1thread": round(m / t_one, 2), "full_graph_s_estimate": round(t_all, 1),
            "full_graph_s_estimate_1thread": round(t_one, 1), "rel_se": round(allc["work_rel_se"], 4),
            "rel_se_1thread": round(one["work_rel_se"], 4), "open_s": round(t_open, 2),
            "sample": f"labelled extrapolation to all {m} edges: the {heaviest} heaviest edges by work proxy "
                      f"(d_u+d_v+sum of neighbour degrees) in full plus a seeded sample (seed {CPU_SEED}) of "
                      f"{n_sample - len(strata[0][2])} edges over {len(strata) - 1} log2-proxy strata, "
                      f"n_h proportional to stratum work; every edge timed; Horvitz-Thompson sum + graph "
                      f"preparation; all cores timed {allc['edges_timed']} edges in {allc['sample_wall_s']:.1f} s, "
                      f"one thread every {thin}th ({one['edges_timed']} edges) in {one['sample_wall_s']:.1f} s"}


def run_reference(args):
    """Reference arm: the CPU oracle on the host cores.  Each step times the
    all-cores stratified sample of cpu_baseline and extrapolates the full
    graph's time; value = edges / the mean extrapolated time."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import graphgen
    import oracle
    g = graphgen.workload(args.workload)
    m = g["m"]
    _, _, proxy = edge_cost_proxy(g)
    full = m <= 20_000                                  # small graphs: every edge timed, as in cpu_baseline
    strata = oracle_design(proxy, m if full else 1000)
    t = time.perf_counter()
    og = oracle.OpenGraph(g)
    t_open = time.perf_counter() - t
    cores = oracle.max_threads()
    for _ in range(args.warmup):
        oracle_estimate(og, strata, cores)
    ests, walls, ses = [], [], []
    for _ in range(args.steps):
        r = oracle_estimate(og, strata, cores)
        ests.append(t_open + r["work_thread_s"] / cores)
        walls.append(r["sample_wall_s"])
        ses.append(r["work_rel_se"])
    one = oracle_estimate(og, strata, 1, thin=1 if full else 10)
    og.close()
    t_full = float(np.mean(ests))
    value = m / t_full
    n_sample = sum(len(x[2]) for x in strata)
    line = {"impl": "reference", "metric": METRIC, "value": round(value, 2), "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(1e3 * float(np.mean(walls)), 3),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int64", "data": "synthetic",
            "config": {"workload": args.workload, "description": WORKLOADS[args.workload], "edges": m,
                       "types": g["L"], "k": 4,
                       "step": "the oracle (Alg. 1-3 + Lemmas, OpenMP over edges) on the stratified edge sample; "
                               "value = edges / extrapolated full-graph time"},
            "cpu_baseline": {"value": round(value, 2), "unit": UNIT, "cores": cores, "kind": "oracle",
                             "value_1thread": round(m / (t_open + one["work_thread_s"]), 2),
                             "full_graph_s_estimate": round(t_full, 1),
                             "step_estimates_spread": round((max(ests) - min(ests)) / t_full, 4),
                             "rel_se": round(float(np.mean(ses)), 4), "open_s": round(t_open, 2),
                             "sample": f"per step: the 100 heaviest edges plus {n_sample - len(strata[0][2])} "
                                       f"seeded edges over {len(strata) - 1} log2-proxy strata (seed {CPU_SEED}), "
                                       f"every edge timed, extrapolated to all {m} edges (same estimator as "
                                       f"the GPU arm's cpu_baseline)"},
            "e2e": {"value": round(value, 2), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def cpu_baseline_sample(graph_of, gpu_totals_of, ids, sizes, seconds: float) -> dict:
    """The CPU-baseline leg of the batched and served forms: the oracle
    (Alg. 1-3 + Lemmas, OpenMP over edges, Sec. 4.7) timed on a seeded
    sample of the graphs (requests), taken smallest first until `seconds`
    of oracle time are spent (0: the whole sample).  The same pass checks
    that each sampled graph's GPU totals equal the oracle's (Sec. 6)."""
    import oracle
    order = sorted(range(len(ids)), key=lambda k: (sizes[k], ids[k]))
    checked, mismatched, edges, spent, largest = 0, [], 0, 0.0, 0
    for k in order:
        if seconds and spent >= seconds:
            break
        x = ids[k]
        g = graph_of(x)
        t = time.perf_counter()
        _, gl = oracle.paper(g, k=4, per_edge=False)
        spent += time.perf_counter() - t
        checked += 1
        edges += g["m"]
        largest = max(largest, g["m"])
        if not np.array_equal(gl, gpu_totals_of(x)):
            mismatched.append(int(x))
    return {"value": round(edges / spent, 1) if spent > 0 else None, "unit": UNIT, "cores": oracle.max_threads(),
            "kind": "oracle",
            "sample": f"{checked} of {len(ids)} seeded sampled graphs ("
                      + ("smallest first within the time budget" if seconds else "all") + f"), {edges} edges, "
                      f"largest {largest} edges, {spent:.1f} s; whole graphs, all 3- and 4-node orbits",
            "totals_identical_to_oracle": not mismatched, "mismatched": mismatched[:20]}


# ------------------------------------------------------------ batched form

def run_batched(args):
    """Batched form: the ego-network batch (graphs with log-uniform edge
    counts 100..400,000, L = 6) as one batch handle counted by one captured
    CUDA graph (tg_count_batch), against plain launches of the same graphs
    one at a time (tg_build + tg_count per graph).  Both produce per-graph
    global totals, which must be identical.  value = edges / time of the
    counting calls (handles built beforehand); build times reported apart."""
    import torch

    import graphgen
    import paper_2010_14058_gb300 as tg
    from paper_2010_14058_gb300 import build as tgbuild
    torch.cuda.set_device(0)
    tgbuild.build()
    def log(msg):
        print(f"[batched] {msg}", file=sys.stderr, flush=True)

    t = time.perf_counter()
    u = graphgen.ego_batch(args.graphs)
    gen_s = time.perf_counter() - t
    log(f"generated {args.graphs} graphs, {u['m']} edges in {gen_s:.1f} s")
    L, m, ng = u["L"], u["m"], args.graphs
    lay = tg.tg_layout(L, 4)
    G = lay["global_slots"]
    stream = torch.cuda.Stream()
    dev = torch.device("cuda")
    rp = torch.as_tensor(u["row_ptr"], device=dev)
    col = torch.as_tensor(u["col"], device=dev)
    ty = torch.as_tensor(u["types"], device=dev)
    torch.cuda.synchronize()
    # autotuned knobs, measured on a sub-batch of the first graphs
    tuned = None
    if args.tune_graphs > 0:
        from paper_2010_14058_gb300 import autotune
        k = min(args.tune_graphs, ng)
        no = u["node_off"]
        nk, zk = int(no[k]), int(u["row_ptr"][int(no[k])])
        t = time.perf_counter()
        tuned = autotune.tune(rp[:nk + 1], col[:zk], ty[:nk], L, node_off=no[:k + 1], reps=1, store=False,
                              stream=stream)
        tuned["tune_s"] = round(time.perf_counter() - t, 1)
        tuned["sub_batch_graphs"] = k
        log(f"autotune on {k} graphs: {tuned['options']} ({tuned['default_ms']} -> {tuned['ms']} ms)")
    options = tuned["options"] if tuned else None
    # batched: one handle, one captured graph
    t = time.perf_counter()
    h = tg.tg_build_batch(u["node_off"], rp, col, ty, L, options=options, stream=stream)
    torch.cuda.synchronize()
    build_batch_s = time.perf_counter() - t
    gl_b = torch.zeros((ng, G), dtype=torch.int64, device=dev)
    with torch.cuda.stream(stream):
        for _ in range(max(args.warmup, 1)):
            tg.tg_count_batch(h, 4, None, gl_b, stream=stream)
        stream.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(args.steps):
            tg.tg_count_batch(h, 4, None, gl_b, stream=stream)
        e1.record(stream)
        stream.synchronize()
    batch_ms = e0.elapsed_time(e1) / args.steps
    log(f"batched: build {build_batch_s:.2f} s, count {batch_ms:.1f} ms")
    launches_batch = h.last_launch_count
    status_b = tg.tg_query_status(h)
    h.free()
    # plain: graph by graph
    gl_p = torch.zeros((ng, G), dtype=torch.int64, device=dev)
    plain_ms, build_plain_s = 0.0, 0.0
    node_off = u["node_off"]
    rp_h = u["row_ptr"]
    status_p = 0
    with torch.cuda.stream(stream):
        for x in range(ng):
            a, b = int(node_off[x]), int(node_off[x + 1])
            s0, s1 = int(rp_h[a]), int(rp_h[b])
            t = time.perf_counter()
            hx = tg.tg_build(rp[a:b + 1] - s0, col[s0:s1] - a, ty[a:b], L, stream=stream)
            stream.synchronize()
            build_plain_s += time.perf_counter() - t
            e0.record(stream)
            tg.tg_count(hx, 4, None, gl_p[x], stream=stream)
            e1.record(stream)
            stream.synchronize()
            plain_ms += e0.elapsed_time(e1)
            status_p = status_p or tg.tg_query_status(hx)
            hx.free()
            if x % 512 == 511:
                log(f"plain: {x + 1} graphs, build {build_plain_s:.1f} s, count {plain_ms:.0f} ms")
    identical = bool(torch.equal(gl_b, gl_p))
    # CPU baseline: the oracle on a seeded 2% sample of the graphs, which
    # also checks their totals
    rng = np.random.default_rng(CPU_SEED + 4)
    k_s = max(1, int(np.ceil(args.oracle_fraction * ng)))
    sample = np.sort(rng.choice(ng, size=min(k_s, ng), replace=False))
    gl_b_h = gl_b.cpu().numpy()

    def graph_of(x):
        a, b = int(node_off[x]), int(node_off[x + 1])
        s0, s1 = int(rp_h[a]), int(rp_h[b])
        return {"n": b - a, "m": (s1 - s0) // 2, "L": L, "row_ptr": rp_h[a:b + 1] - s0,
                "col": u["col"][s0:s1] - a, "types": u["types"][a:b]}

    cpu = cpu_baseline_sample(graph_of, lambda x: gl_b_h[x], sample.tolist(),
                              [int(u["graph_m"][x]) for x in sample], args.oracle_seconds)
    log(f"oracle sample: {cpu}")
    line = {"metric": METRIC + ", batched form", "value": round(m / (batch_ms / 1e3), 1), "unit": UNIT, "n_gpus": 1,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(batch_ms, 3), "higher_is_better": True,
            "dtype": "int64", "data": "synthetic",
            "config": {"workload": f"ego_batch({ng})", "graphs": ng, "edges": m, "nodes": u["n"], "types": L,
                       "graph_edges_median": float(np.median(u["graph_m"])), "graph_edges_max": int(u["graph_m"].max()),
                       "parent": "Chung-Lu n=4e6 m=4e7 gamma=2.3 max weight 2e4", "generation_s": round(gen_s, 1)},
            "batched": {"count_ms": round(batch_ms, 3), "edges_per_s": round(m / (batch_ms / 1e3), 1),
                        "build_s": round(build_batch_s, 3), "launches_per_count": launches_batch,
                        "status": tg.STATUS[status_b],
                        "autotune": None if tuned is None else {x: tuned[x] for x in (
                            "options", "default_ms", "ms", "sub_batch_graphs", "tune_s", "signature")}},
            "plain_per_graph": {"count_ms": round(plain_ms, 3), "edges_per_s": round(m / (plain_ms / 1e3), 1),
                                "build_s": round(build_plain_s, 3), "status": tg.STATUS[status_p]},
            "speedup_count": round(plain_ms / batch_ms, 2),
            "speedup_build_plus_count": round((build_plain_s + plain_ms / 1e3) / (build_batch_s + batch_ms / 1e3), 2),
            "totals_identical": identical, "cpu_baseline": cpu}
    print(json.dumps(line), flush=True)


# -------------------------------------------------------------- serving

def run_serve(args):
    """Serving form: open-loop Poisson arrivals of typed graphs (Chung-Lu
    gamma = 2.2, edges log-uniform in [100, 1e6], n = m/5, L uniform 3..8)
    drawn from a seeded pool, for a warm-up and then the measured window;
    served with admission by a 40 GB device budget, micro-batching and 4
    overlapped workers, with and without 16 GB of resident handles.  The
    plain sequential server (one worker, no micro-batching, the same resident
    cache) replays the trace up to warm-up + plain_seconds.  Reports p50/p99
    latency and sustained edges/s of each over its measured window, and
    whether every result is identical."""
    import torch

    from paper_2010_14058_gb300 import build as tgbuild
    from paper_2010_14058_gb300 import serve
    torch.cuda.set_device(0)
    tgbuild.build()

    def log(msg):
        print(f"[serve] {msg}", file=sys.stderr, flush=True)

    t = time.perf_counter()
    pool = serve.request_pool(args.pool, seed=20201029 + 5)
    gen_s = time.perf_counter() - t
    w0 = args.serve_warmup
    trace = serve.poisson_trace(pool, args.rate, w0 + args.duration, seed=20201029 + 5)
    log(f"pool of {len(pool)} graphs in {gen_s:.1f} s; {len(trace)} requests, "
        f"{sum(r.m for r in trace)} edges")
    serve.Server(workers=4).run(serve.poisson_trace(pool, 200.0, 0.2, seed=1))      # first launches, pool
    runs = {}
    for name, resident in (("served", 16 << 30), ("served_no_resident", 0)):
        t = time.perf_counter()
        srv = serve.Server(budget_bytes=40 << 30, workers=4, resident_bytes=resident)
        runs[name] = srv.run(trace)
        srv.close()
        log(f"{name}: {time.perf_counter() - t:.1f} s")
    prefix = [r for r in trace if r.arrival < w0 + args.plain_seconds]
    t = time.perf_counter()
    srv = serve.Server(budget_bytes=40 << 30, workers=1, batching=False, resident_bytes=16 << 30)
    plain = srv.run(prefix)
    srv.close()
    log(f"plain sequential on {len(prefix)} requests: {time.perf_counter() - t:.1f} s")
    by_rid = {name: {r.rid: r for r in res} for name, res in runs.items()}
    same = all(r.status == 0 for res in runs.values() for r in res) and all(r.status == 0 for r in plain)
    same = same and all(np.array_equal(a.totals, by_rid["served_no_resident"][a.rid].totals) for a in runs["served"])
    same = same and all(np.array_equal(p.totals, by_rid["served"][p.rid].totals) for p in plain)
    # CPU baseline: the oracle on a seeded 2% sample of the requests, which
    # also checks their totals
    rng = np.random.default_rng(CPU_SEED + 5)
    k_s = max(1, int(np.ceil(args.oracle_fraction * len(trace))))
    sample = np.sort(rng.choice(len(trace), size=min(k_s, len(trace)), replace=False)).tolist()

    def request_graph(x):
        r = trace[x]
        return {"n": r.n, "m": r.m, "L": r.L, "row_ptr": r.row_ptr, "col": r.col, "types": r.types}

    cpu = cpu_baseline_sample(request_graph, lambda x: by_rid["served"][trace[x].rid].totals, sample,
                              [trace[x].m for x in sample], args.oracle_seconds)
    summ = {name: serve.summarize(res, trace, window_start=w0) for name, res in runs.items()}
    s0 = serve.summarize(plain, prefix, window_start=w0)
    line = {"metric": METRIC + ", serving form", "value": summ["served"]["edges_per_s"], "unit": UNIT, "n_gpus": 1,
            "higher_is_better": True, "dtype": "int64", "data": "synthetic",
            "config": {"workload": "poisson_requests", "rate_per_s": args.rate, "warmup_seconds": w0,
                       "arrival_seconds": args.duration, "requests": len(trace),
                       "edges": int(sum(r.m for r in trace)), "pool_graphs": args.pool,
                       "request_mix": "Chung-Lu gamma=2.2, m log-uniform [100, 1e6], n=m/5, L uniform 3..8",
                       "budget_gb": 40, "resident_gb": 16, "workers": 4, "pool_generation_s": round(gen_s, 1),
                       "plain_sequential_trace": f"arrivals before {w0 + args.plain_seconds:.0f} s "
                                                 f"({len(prefix)} requests), one worker, no micro-batching, "
                                                 f"the same 16 GB resident cache"},
            "served": summ["served"], "served_no_resident": summ["served_no_resident"], "plain_sequential": s0,
            "results_identical": bool(same), "cpu_baseline": cpu}
    print(json.dumps(line), flush=True)


if __name__ == "__main__":
    a = parse()
    if a.mode == "serve" and a.impl != "reference":
        run_serve(a)
        sys.exit(0)
    if a.impl == "reference":
        run_reference(a)
    elif a.mode == "batched":
        run_batched(a)
    else:
        run_ours(a)
