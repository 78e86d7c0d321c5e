#!/usr/bin/env python3
"""Benchmark of the GB300 GGArray on the paper-shaped growth workload.

One step is one pass of the whole hot path over one batch of synthetic input
(1024 blocks x 512 threads, first bucket 4096 int32 elements):

  clear (buckets back to the free lists) -> gga_insert of 512 rounds of
  Uniform{0,1,2} per-thread insertions (~2^28 elements, 1 GiB) -> 2^26
  random-index reads -> 2^26 random-index writes -> rw_b +1 sweep -> rw_g +1
  sweep -> flatten into a contiguous array.

`value` is elements inserted per second of step time (Gelem/s), inputs
resident in HBM (larger than L2, so no flush is needed).  `e2e` repeats the
step through the same C-ABI calls with the inputs copied from pinned host
memory each step and the read results and the flattened array copied back.
With torchrun, every rank grows its own replica (weak scaling, no data-path
collective); the time is the max over ranks.

`--impl reference` times the CPU oracle on a bounded sample of the same
workload instead (rank 0 only).
"""

from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np
import torch

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "GGArray insert Gelem/s & % HBM roofline; mem/needed; served p99 latency"
PEAKS_FALLBACK = {"hbm_gbs": 6800.0}
# Kernels per phase: a write batch of 2^20 or more goes through bins (count,
# scan, scatter into bins, apply), a smaller one is one kernel; a read batch of
# 2^25 or more from a slab of at most 48 bytes per read goes through bins too
# (decide, count, scatter, apply, return).  An insertion of up to 1024 count
# tiles (32 rows each at T = 512) scans them in its count kernel.
LAUNCHES_PER_STEP = {"clear": 1, "insert": 4, "read": 5, "write": 4, "rw_b": 1, "rw_g": 1, "flatten": 1}
BINNED_WRITE_MIN = 1 << 20
BINNED_READ_MIN = 1 << 25
BINNED_READ_SLAB = (512 << 20, 48)   # bytes at least, bytes per read at most


def launches_per_step(n_rand: int, slab_bytes: int, rows: int) -> int:
    n = sum(LAUNCHES_PER_STEP.values())
    if n_rand < BINNED_WRITE_MIN:
        n -= 3
    if not read_is_binned(n_rand, slab_bytes):
        n -= 4
    return n - (1 if rows <= 32 * 1024 else 0)


def read_is_binned(n_rand: int, slab_bytes: int) -> bool:
    least, per_read = BINNED_READ_SLAB
    return n_rand >= BINNED_READ_MIN and slab_bytes >= least and slab_bytes // per_read <= n_rand


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--rounds", type=int, default=512, help="insertion rounds per step (512 = full workload)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-baselines", action="store_true", help="skip the static / semi-static flat arrays")
    ap.add_argument("--nvtx", action="store_true", help="NVTX range around every phase of a step (for a profiler)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--e2e-steps", type=int, default=None,
                    help="steps of the end-to-end loop (default: --steps, as the device-timed loop)")
    ap.add_argument("--workload", choices=["paper_growth", "batched", "served", "two_phase", "doubling",
                                           "insertion", "phases", "random_access"],
                    default="paper_growth",
                    help="paper_growth: the headline step; batched: 4096 arrays in one persistent launch; "
                         "served: continuous-batching request server")
    ap.add_argument("--duration", type=float, default=10.0, help="served: seconds of offered load")
    ap.add_argument("--newborn", action="store_true", help="two_phase: only the previous generation spawns")
    ap.add_argument("--arrays", type=int, default=4096, help="batched: number of arrays (a smaller case for profiling)")
    ap.add_argument("--n0", type=int, default=1 << 24, help="two_phase: initial records (a smaller case for profiling)")
    ap.add_argument("--generations", type=int, default=8, help="two_phase: spawning generations")
    ap.add_argument("--no-sweep", action="store_true", help="served: skip the arrival-rate sweep")
    ap.add_argument("--l2-fetch", type=int, default=0,
                    help="random_access: the context's L2 fetch granularity hint in bytes (0: leave the default)")
    ap.add_argument("--deadline", type=float, default=None,
                    help="served: seconds an append may wait for pool memory before it is rejected")
    return ap.parse_args()


# Source files that define each kernel: a recorded DRAM traffic figure is
# only used while their hash matches the one stored with it.
SECTOR_BYTES = 32   # DRAM/L2 sector: the least a random element access moves
DEVICE_H = "include/gga_layout.cuh"
KERNEL_SOURCES = {
    "write_kernel": ["gga_access.cu", "gga_core.cuh", DEVICE_H],
    "read_kernel": ["gga_access.cu", "gga_core.cuh", DEVICE_H],
    "flatten_kernel": ["gga_access.cu", "gga_core.cuh", DEVICE_H],
    "sweep_b_kernel": ["gga_access.cu", "gga_core.cuh", DEVICE_H],
    "sweep_g_kernel": ["gga_access.cu", "gga_core.cuh", DEVICE_H],
    "copy_bulk_kernel": ["gga_insert.cu", "gga_core.cuh", "gga_gen.cuh", DEVICE_H],
    "count_kernel": ["gga_insert.cu", "gga_core.cuh", "gga_gen.cuh", DEVICE_H],
    "wbin_count_kernel": ["gga_access.cu", "gga_core.cuh", DEVICE_H],
    "wbin_scatter_kernel": ["gga_access.cu", "gga_core.cuh", DEVICE_H],
    "wbin_apply_kernel": ["gga_access.cu", "gga_core.cuh", DEVICE_H],
}
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "dram_traffic_per_kernel_paper_growth_R96.md")


def kernel_source_path(f: str) -> str:
    """A KERNEL_SOURCES entry: a path from the repository root for the public
    headers, else a file of the package's csrc/."""
    return os.path.join(ROOT, f) if f.startswith("include/") else os.path.join(ROOT, "paper_2209_00103_gb300", "csrc", f)


def kernel_source_sha(kernel: str) -> str:
    import hashlib
    h = hashlib.sha256()
    for f in KERNEL_SOURCES.get(kernel, []):
        with open(kernel_source_path(f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:12]


def recorded_traffic(kernel: str, units: int):
    """DRAM bytes of one launch of `kernel` over `units` work units (reads,
    writes, elements or count rows, as the kernel's row of the committed
    table says), from one-kernel ncu captures of the 96-round case scaled by
    units / captured units; None if the kernel has no row or its source
    changed since the capture."""
    try:
        for line in open(TRAFFIC_FILE):
            cells = [c.strip() for c in line.strip().strip("|").split("|")]
            if len(cells) >= 6 and cells[0] == kernel and cells[5] == kernel_source_sha(kernel):
                return int(round(int(cells[4]) * units / int(cells[3])))
    except (OSError, ValueError, ZeroDivisionError):
        pass
    return None


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return PEAKS_FALLBACK["hbm_gbs"], "fallback"


# ---------------------------------------------------------------------------
# Distributed plumbing (one process per GPU; no data-path collective).

def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        backend = "nccl" if torch.cuda.is_available() else "gloo"
        if torch.cuda.is_available():
            torch.cuda.set_device(local)
        dist.init_process_group(backend=backend)
    elif torch.cuda.is_available():
        torch.cuda.set_device(local)
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x: float, world: int) -> float:
    if world == 1:
        return x
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def sum_over_ranks(x: float, world: int) -> float:
    if world == 1:
        return x
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


# ---------------------------------------------------------------------------
# Clock sampling during the timed region.

class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(prefix="gga_clocks_", suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits", "-lms", "50",
                 "-i", str(self.gpu)], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
            time.sleep(0.3)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.1)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = []
        try:
            for line in open(self.path):
                parts = [p.strip() for p in line.split(",")]
                if len(parts) >= 9 and parts[1].replace(".", "").isdigit():
                    rows.append(parts)
            os.unlink(self.path)
        except Exception:
            pass
        if not rows:
            return None
        sm = [float(r[1]) for r in rows]
        mx = [float(r[2]) for r in rows]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        try:
            pw = max(float(r[3]) for r in rows)
        except ValueError:
            pw = None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": reasons,
                "samples": len(rows), "power_w_max": pw}


# ---------------------------------------------------------------------------
# The GPU arm.

def algorithmic_bytes(N, R, L, T, E, n_rand):
    """Bytes each phase must move at minimum: insertion reads the R*L*T
    4-byte counts and the N packed values and writes the N elements; a
    random read or write moves its 8-byte index, the element and the
    output (or input) value; sweeps and flatten read and write every
    element once."""
    counts = R * L * T * 4
    return {
        "insert": counts + 2 * N * E,          # counts read, values read, elements written
        "read": n_rand * (8 + E + E),          # index, element, output
        "write": n_rand * (8 + E + E),         # index, input, element
        "rw_b": 2 * N * E,
        "rw_g": 2 * N * E,
        "flatten": 2 * N * E,
    }


def run_ours(args, world, rank, local):
    from paper_2209_00103_gb300 import gga
    from paper_2209_00103_gb300 import workloads as wl

    w = wl.paper_growth()
    R = args.rounds
    spec = wl.InsertSpec(L=w.L, T=w.T, E=w.E, seed=w.spec.seed + 1000 * rank, dist=w.spec.dist, rounds=R,
                         coeffs=w.spec.coeffs)
    dev = torch.device("cuda", local)
    counts, values = wl.make_insert_inputs_t(spec, dev)
    N = int(values.shape[0])
    n_rand = w.n_random if R == 512 else max(1, w.n_random * R // 512)
    idx_r = wl.uniform_indices_t(w.read_seed, n_rand, N, dev)
    idx_w = wl.uniform_indices_t(w.write_seed, n_rand, N, dev)
    vals_w = wl.index_keyed_values_t(w.value_seed, idx_w, w.E)
    out_r = gga.elem_tensor(n_rand, w.E, dev)
    dst = gga.elem_tensor(N, w.E, dev)
    pool_bytes = int(2.5 * N * w.E) + w.L * w.B * w.E * 4
    g = gga.GGArray(w.L, w.T, w.B, w.E, pool_bytes)
    stream = torch.cuda.current_stream(dev)

    phases = ["clear", "insert", "read", "write", "rw_b", "rw_g", "flatten"]

    nvtx = torch.cuda.nvtx if args.nvtx else None

    def step(ev=None):
        def mark(i):
            if ev is not None:
                ev[i].record(stream)
            if nvtx is not None:
                if i > 0:
                    nvtx.range_pop()
                if i < len(phases):
                    nvtx.range_push(phases[i])
        mark(0)
        g.clear(stream)
        mark(1)
        g.insert(counts, values, stream)
        mark(2)
        g.read(idx_r, out_r, stream)
        mark(3)
        g.write(idx_w, vals_w, stream)
        mark(4)
        g.sweep(gga.GGA_RW_B, 1, 1, stream)
        mark(5)
        g.sweep(gga.GGA_RW_G, 1, 1, stream)
        mark(6)
        g.flatten(dst, stream)
        mark(7)

    for _ in range(max(3, args.warmup)):
        step()
    torch.cuda.synchronize(dev)
    n_check, rc = g.size(stream)
    if rc != gga.GGA_OK or n_check != N:
        raise RuntimeError(f"warm-up step failed: size {n_check} vs {N}, device error {rc}")
    mem = g.memory(stream)

    K = args.steps
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(8)] for _ in range(K)]
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    sampler = ClockSampler(local)
    barrier(world)
    torch.cuda.synchronize(dev)
    sampler.start()
    t0.record(stream)
    for k in range(K):
        step(evs[k])
    t1.record(stream)
    torch.cuda.synchronize(dev)
    clocks = sampler.stop()
    barrier(world)
    elapsed_ms = t0.elapsed_time(t1)
    if g.last_error(stream) != gga.GGA_OK:
        raise RuntimeError("device error during the timed steps")
    t_max_ms = max_over_ranks(elapsed_ms, world)
    total_elems = sum_over_ranks(float(N * K), world)
    value = total_elems / (t_max_ms / 1e3) / 1e9

    # Per-phase device times (ms, median over steps).
    ph_ms = {}
    for i, name in enumerate(phases):
        ph_ms[name] = statistics.median(evs[k][i].elapsed_time(evs[k][i + 1]) for k in range(K))
    peak, peak_src = peaks()
    ab = algorithmic_bytes(N, R, w.L, w.T, w.E, n_rand)
    phase_info = {}
    for name in phases:
        d = {"ms": round(ph_ms[name], 4)}
        if name in ab:
            gbs = ab[name] / (ph_ms[name] / 1e3) / 1e9
            d.update({"algorithmic_bytes": ab[name], "achieved_gbs": round(gbs, 1),
                      "frac_of_measured_peak": round(gbs / peak, 3), "frac_of_8tbs": round(gbs / 8000.0, 3)})
        if name == "insert":
            d["gelem_s"] = round(N / (ph_ms[name] / 1e3) / 1e9, 2)
        if name in ("read", "write"):
            # Sector-effective: an element access moves at least one 32-byte
            # sector, so each access counts index + sector + the other side.
            sec = n_rand * (8 + SECTOR_BYTES + w.E)
            d["sector_effective_gbs"] = round(sec / (ph_ms[name] / 1e3) / 1e9, 1)
            d["sector_effective_frac"] = round(sec / (ph_ms[name] / 1e3) / 1e9 / peak, 3)
        phase_info[name] = d

    # The dominant kernel carries the roofline record: the longest phase that
    # is one kernel (insert and binned reads and writes are several; the launch
    # list in profiles/ confirms which single kernel takes the most time).
    binned = n_rand >= BINNED_WRITE_MIN
    binned_read = read_is_binned(n_rand, pool_bytes)
    single = ["flatten", "rw_b", "rw_g"] + ([] if binned_read else ["read"]) + ([] if binned else ["write"])
    dom = max(single, key=lambda n: ph_ms[n])
    kernels = {"insert": "count_kernel + tile_scan_kernel + reserve_kernel + copy_bulk_kernel",
               "flatten": "flatten_kernel", "rw_b": "sweep_b_kernel", "rw_g": "sweep_g_kernel",
               "read": ("rbin_decide_kernel + rbin_count_kernel + rbin_scatter_kernel + rbin_apply_kernel + "
                        "rbin_return_kernel" if binned_read else "read_kernel"),
               "write": ("wbin_count_kernel + wbin_scan_kernel + wbin_scatter_kernel + wbin_apply_kernel"
                         if binned else "write_kernel")}
    for name in ("insert", "read", "write"):
        phase_info[name]["kernels"] = kernels[name]
    ach = ab[dom] / (ph_ms[dom] / 1e3) / 1e9
    units = {"read": n_rand, "write": n_rand, "flatten": N, "rw_b": N, "rw_g": N}
    traffic = recorded_traffic(kernels[dom], units[dom]) if dom in units else None
    roofline = {"bound": "hbm", "achieved": round(ach, 1), "peak": peak, "unit": "GB/s",
                "frac": round(ach / peak, 3), "traffic": traffic, "kernel": kernels[dom], "phase": dom,
                "algorithmic_bytes_per_launch": ab[dom],
                "peak_source": f"{peak_src} (MEASURED_PEAKS.json hbm_gbs)" if peak_src == "measured" else peak_src}
    if traffic:
        roofline["traffic_gbs"] = round(traffic / (ph_ms[dom] / 1e3) / 1e9, 1)
    # Insert carries the headline roofline of the growable array itself.
    ins_gbs = ab["insert"] / (ph_ms["insert"] / 1e3) / 1e9

    # The paper's comparison arrays (Sec. II) on the same inputs.
    baselines = None
    if not args.no_baselines and rank == 0 and w.E == 4:
        baselines = run_flat_baselines(counts, values, idx_r, idx_w, vals_w, N, R, w.L, w.T, dev, stream)
        if dom == "read" or binned_read:
            # A random gather is bound by the DRAM access rate, not by its
            # bytes: the same indices gathered from a flat int32 array by
            # PyTorch (grouped by ranges first, the read phase passes it).
            flat_ms = baselines["static"]["phases_ms"]["read"]
            (roofline if dom == "read" else phase_info["read"])["vs_flat_gather"] = {
                "flat_ms": flat_ms, "ms": round(ph_ms["read"], 4), "frac": round(flat_ms / ph_ms["read"], 3),
                "accesses_per_s": round(n_rand / (ph_ms["read"] / 1e3) / 1e9, 2), "unit": "G accesses/s",
                "flat": "torch.index_select on a flat int32 array of the same size, same indices"}

    # End to end through the C ABI with host buffers.
    e2e = None
    if not args.no_e2e:
        e2e = run_e2e(args, g, counts, values, idx_r, idx_w, vals_w, out_r, dst, N, world, dev, stream)

    # In-kernel generated insertion (values drawn by the inserting threads):
    # rounds batched in passes, and the device API's one push per round.
    gen = time_generated(w, R, pool_bytes, dev, stream)
    push_gen = time_generated(w, R, pool_bytes, dev, stream, per_round=True)
    push_exp = time_push_expand(spec, w.B, counts, pool_bytes, dev, stream)

    result = {
        "metric": METRIC, "value": round(value, 3), "unit": "Gelem/s", "n_gpus": world, "steps": K,
        "warmup": max(3, args.warmup), "ms_per_step": round(t_max_ms / K, 4), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
        "config": {"workload": f"paper_growth_{w.L}x{w.T}_B{w.B}_int32_R{R}", "L": w.L, "T": w.T, "B": w.B,
                   "elem_bytes": w.E, "rounds": R, "count_dist": "uniform{0,1,2}", "elements_per_gpu": N,
                   "random_reads": n_rand, "random_writes": n_rand,
                   "step": "clear+insert(all rounds, one call)+read+write+rw_b(+1)+rw_g(+1)+flatten",
                   "l2": "inputs larger than L2 (counts and values 1 GiB each), no flush",
                   "parallelism": f"replicas x{world}"},
        "roofline": roofline,
        "insert_roofline": {"achieved": round(ins_gbs, 1), "peak": peak, "unit": "GB/s",
                            "frac": round(ins_gbs / peak, 3), "frac_of_8tbs": round(ins_gbs / 8000.0, 3),
                            "gelem_s": phase_info["insert"]["gelem_s"]},
        "phases": phase_info,
        "mem_over_needed": round(mem["bucket_bytes"] / max(1, mem["live_bytes"]), 4),
        "memory": mem,
        "insert_generated": gen,
        "push_generated": push_gen,
        "push_expand": push_exp,
        "gpu_launches": K * launches_per_step(n_rand, pool_bytes, R * w.L),
        "clocks": clocks,
        "e2e": e2e,
        "baselines": baselines,
    }
    if rank == 0 and not args.no_cpu_baseline:
        result["cpu_baseline"] = cpu_baseline(R)
    g.close()
    return result


def run_flat_baselines(counts, values, idx_r, idx_w, vals_w, N, R, L, T, dev, stream, steps=5):
    """The comparison arrays of the paper's Sec. II on the same inputs and GPU,
    as plain flat arrays with PyTorch's own kernels (they are baselines, not
    part of the GGArray path):
      static       allocated once for the worst case (every thread inserting 2
                   elements every round), so no growth ever happens;
      semi_static  grown from the host by doubling: before each round the
                   host reads the round's total (one synchronization) and, if
                   it does not fit, allocates twice the capacity and copies.
    Values arrive packed in prefix-sum order, so an insertion writes them
    contiguously after the current size.  A flat array is already
    contiguous: it needs no flatten.  Both sweeps (rw_b, rw_g) are one +1 pass."""
    per_round = counts.view(R, -1)
    out = {}

    def phase_times(run, k):
        names = ["insert", "read", "write", "rw_b", "rw_g"]
        res = {n: [] for n in names}
        for _ in range(k):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(len(names) + 1)]
            run(ev)
            torch.cuda.synchronize(dev)
            for i, n in enumerate(names):
                res[n].append(ev[i].elapsed_time(ev[i + 1]))
        return {n: round(statistics.median(v), 4) for n, v in res.items()}

    read_out = torch.empty_like(idx_r, dtype=values.dtype)

    # Static: worst-case capacity.
    cap = 2 * R * L * T
    a = torch.empty(cap, dtype=values.dtype, device=dev)

    def static_step(ev):
        ev[0].record(stream)
        total = per_round.sum()                            # the insertion's size update (< 2^31 here)
        a[:N].copy_(values)
        ev[1].record(stream)
        torch.index_select(a[:N], 0, idx_r, out=read_out)
        ev[2].record(stream)
        a.index_copy_(0, idx_w, vals_w)
        ev[3].record(stream)
        a[:N].add_(1)
        ev[4].record(stream)
        a[:N].add_(1)
        ev[5].record(stream)
        return total

    phase_times(static_step, 2)
    ph = phase_times(static_step, steps)
    ms = sum(ph.values())
    out["static"] = {"capacity_elems": cap, "mem_over_needed": round(cap / N, 4), "phases_ms": ph,
                     "flatten_ms": 0.0, "ms_per_step": round(ms, 4), "gelem_s": round(N / (ms / 1e3) / 1e9, 3)}
    del a

    # Semi-static: host-resized by doubling, checked every round.
    state = {}

    def semi_step(ev):
        ev[0].record(stream)
        c = 1 << 20
        buf = torch.empty(c, dtype=values.dtype, device=dev)
        size = 0
        for r in range(R):
            n_r = int(per_round[r].sum().item())                   # host learns the round's total
            if size + n_r > c:
                while size + n_r > c:
                    c *= 2
                nb = torch.empty(c, dtype=values.dtype, device=dev)
                nb[:size].copy_(buf[:size])
                buf = nb
            buf[size:size + n_r].copy_(values[size:size + n_r])
            size += n_r
        ev[1].record(stream)
        torch.index_select(buf[:size], 0, idx_r, out=read_out)
        ev[2].record(stream)
        buf.index_copy_(0, idx_w, vals_w)
        ev[3].record(stream)
        buf[:size].add_(1)
        ev[4].record(stream)
        buf[:size].add_(1)
        ev[5].record(stream)
        state["cap"] = c
        state["size"] = size

    phase_times(semi_step, 1)
    ph = phase_times(semi_step, max(1, steps // 2))
    ms = sum(ph.values())
    out["semi_static"] = {"capacity_elems": state["cap"], "mem_over_needed": round(state["cap"] / N, 4),
                          "phases_ms": ph, "flatten_ms": 0.0, "host_syncs_per_step": R,
                          "ms_per_step": round(ms, 4), "gelem_s": round(N / (ms / 1e3) / 1e9, 3)}
    if state["size"] != N:
        raise RuntimeError("semi-static baseline inserted a wrong number of elements")
    out["note"] = ("flat arrays with PyTorch kernels (index_select / index_copy_ / add_); "
                   "the GGArray's write phase uses its own binned writes")
    return out


def run_e2e(args, g, counts, values, idx_r, idx_w, vals_w, out_r, dst, N, world, dev, stream):
    """The step through the C ABI with host buffers: every step copies its
    inputs (counts, values, read and write indices, written values) from
    pinned host memory and copies its results (the random reads and the
    flattened array) back.  Steps are pipelined as a throughput user would
    run them: inputs and outputs are double-buffered on the device, uploads
    run on one copy stream and downloads on another, so step k+1's upload
    and step k-1's download overlap step k's kernels; events order every
    reuse of a buffer."""
    from paper_2209_00103_gb300 import gga
    ins = [counts, values, idx_r, idx_w, vals_w]
    host_in = [t.cpu().pin_memory() for t in ins]
    host_out = [torch.empty(out_r.shape, dtype=out_r.dtype).pin_memory(),
                torch.empty(dst.shape, dtype=dst.dtype).pin_memory()]
    dev_in = [[t, torch.empty_like(t)] for t in ins]             # two sets: the bench's own tensors and a copy
    dev_out = [[out_r, torch.empty_like(out_r)], [dst, torch.empty_like(dst)]]
    h2d = sum(t.numel() * t.element_size() for t in host_in)
    d2h = sum(t.numel() * t.element_size() for t in host_out)
    up = torch.cuda.Stream(dev)
    down = torch.cuda.Stream(dev)
    inputs_free = [None, None]     # compute finished with input set b
    outputs_free = [None, None]    # download finished with output set b

    def event_on(s):
        e = torch.cuda.Event()
        e.record(s)
        return e

    def step(k):
        b = k & 1
        if inputs_free[b] is not None:
            up.wait_event(inputs_free[b])
        with torch.cuda.stream(up):
            for d, h in zip(dev_in, host_in):
                d[b].copy_(h, non_blocking=True)
        ready = event_on(up)
        stream.wait_event(ready)
        if outputs_free[b] is not None:
            stream.wait_event(outputs_free[b])
        g.clear(stream)
        g.insert(dev_in[0][b], dev_in[1][b], stream)
        g.read(dev_in[2][b], dev_out[0][b], stream)
        g.write(dev_in[3][b], dev_in[4][b], stream)
        g.sweep(gga.GGA_RW_B, 1, 1, stream)
        g.sweep(gga.GGA_RW_G, 1, 1, stream)
        g.flatten(dev_out[1][b], stream)
        done = event_on(stream)
        inputs_free[b] = done
        down.wait_event(done)
        with torch.cuda.stream(down):
            host_out[0].copy_(dev_out[0][b], non_blocking=True)
            host_out[1].copy_(dev_out[1][b], non_blocking=True)
        outputs_free[b] = event_on(down)

    for k in range(2):
        step(k)
    torch.cuda.synchronize(dev)

    def copy_gbs(dst, src, s, reps=3):
        best = None
        for _ in range(reps):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(s)
            with torch.cuda.stream(s):
                dst.copy_(src, non_blocking=True)
            e1.record(s)
            torch.cuda.synchronize(dev)
            ms = e0.elapsed_time(e1)
            best = ms if best is None else min(best, ms)
        return src.numel() * src.element_size() / (best / 1e3) / 1e9

    # The host link alone, on the largest input and output of the step: the
    # step cannot run faster than its uploads at this rate.
    h2d_gbs = copy_gbs(dev_in[1][1], host_in[1], up)
    d2h_gbs = copy_gbs(host_out[1], dev_out[1][1], down)
    barrier(world)
    K = args.e2e_steps if args.e2e_steps is not None else args.steps
    a = torch.cuda.Event(enable_timing=True)
    b_ev = torch.cuda.Event(enable_timing=True)
    a.record(stream)
    up.wait_event(a)
    down.wait_event(a)
    for k in range(K):
        step(k)
    stream.wait_event(outputs_free[(K - 1) & 1])
    b_ev.record(stream)
    torch.cuda.synchronize(dev)
    ms = max_over_ranks(a.elapsed_time(b_ev), world)
    total = sum_over_ranks(float(N * K), world)
    for t in dev_in:
        del t[1]
    del dev_out[0][1], dev_out[1][1]
    bound_ms = h2d / (h2d_gbs * 1e9) * 1e3
    return {"value": round(total / (ms / 1e3) / 1e9, 3), "unit": "Gelem/s", "h2d_bytes_per_step": int(h2d),
            "d2h_bytes_per_step": int(d2h), "ms_per_step": round(ms / K, 3), "steps": K,
            "pipelining": "double-buffered inputs/outputs, uploads and downloads on their own streams",
            "host_link": {"h2d_gbs": round(h2d_gbs, 1), "d2h_gbs": round(d2h_gbs, 1),
                          "h2d_bound_ms_per_step": round(bound_ms, 3), "frac": round(bound_ms / (ms / K), 3),
                          "note": "pinned copies of the step's values (h2d) and flattened array (d2h) alone, "
                                  "CUDA events; the bound is the step's uploads at the h2d rate"}}


def time_generated(w, R, pool_bytes, dev, stream, per_round=False):
    """The generated insertion of the workload's rounds: gga_insert_generated
    (rounds batched in passes), or with per_round gga_push_generated (the
    device API: one gga::BlockPusher push per round, Algorithm 1 as written)."""
    from paper_2209_00103_gb300 import gga
    g = gga.GGArray(w.L, w.T, w.B, w.E, pool_bytes)
    spec = gga.make_gen_spec(w.spec.seed, w.spec.dist, w.spec.coeffs)
    run = g.push_generated if per_round else g.insert_generated
    for _ in range(3):
        g.clear(stream)
        run(spec, R, stream)
    torch.cuda.synchronize(dev)
    n, rc = g.size(stream)
    K = 10
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(K)]
    for a, b in evs:
        g.clear(stream)
        a.record(stream)
        run(spec, R, stream)
        b.record(stream)
    torch.cuda.synchronize(dev)
    ms = statistics.median(a.elapsed_time(b) for a, b in evs)
    g.close()
    gbs = n * w.E / (ms / 1e3) / 1e9
    peak, _ = peaks()
    return {"elements": n, "ms": round(ms, 4), "gelem_s": round(n / (ms / 1e3) / 1e9, 2),
            "achieved_gbs": round(gbs, 1), "frac_of_measured_peak": round(gbs / peak, 3),
            "device_error": rc,
            "kernels": ("push_generated_kernel" if per_round else "gen_insert_kernel") + " + finalize_kernel",
            "algorithmic_bytes": "E per element (values drawn in registers, write only)"}


def time_push_expand(spec, B, counts, pool_bytes, dev, stream):
    """Pushes of values read from device memory through the device API
    (gga_push_expand: gga::RoundsPusher, 4 rounds per push): the same
    counts as the step's insertion, and one int32 input per (round, block,
    thread) that the thread appends `count` times.  Algorithmic bytes: the
    counts and inputs read (4 + E per thread and round) and E per element
    written."""
    from paper_2209_00103_gb300 import gga
    from paper_2209_00103_gb300 import workloads as wl
    inputs = wl.expand_inputs_t(spec, dev)
    g = gga.GGArray(spec.L, spec.T, B, spec.E, pool_bytes)
    for _ in range(3):
        g.clear(stream)
        g.push_expand(counts, inputs, stream)
    torch.cuda.synchronize(dev)
    n, rc = g.size(stream)
    K = 10
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(K)]
    for a, b in evs:
        g.clear(stream)
        a.record(stream)
        g.push_expand(counts, inputs, stream)
        b.record(stream)
    torch.cuda.synchronize(dev)
    ms = statistics.median(a.elapsed_time(b) for a, b in evs)
    g.close()
    del inputs
    slots = counts.numel()
    alg = slots * (4 + spec.E) + n * spec.E
    gbs = alg / (ms / 1e3) / 1e9
    peak, _ = peaks()
    return {"elements": n, "ms": round(ms, 4), "gelem_s": round(n / (ms / 1e3) / 1e9, 2),
            "algorithmic_bytes": int(alg), "achieved_gbs": round(gbs, 1), "frac_of_measured_peak": round(gbs / peak, 3),
            "frac_of_8tbs": round(gbs / 8000.0, 3), "device_error": rc,
            "kernels": "push_expand_s_kernel + finalize_kernel",
            "note": "counts [R][L][T] and one input per (round, block, thread) read from HBM; "
                    "RoundsPusher pushes of 4 rounds, 4 slots per thread, loads a push ahead, staged 128-bit stores"}


# ---------------------------------------------------------------------------
# The oracle arms (host cores).

def oracle_sample(rounds: int):
    """One bounded sample step of the workload on the CPU oracle; returns
    (elements inserted, seconds, description)."""
    import oracle
    from paper_2209_00103_gb300 import workloads as wl
    w = wl.paper_growth()
    spec = wl.InsertSpec(L=w.L, T=w.T, E=w.E, seed=w.spec.seed, dist=w.spec.dist, rounds=rounds,
                         coeffs=w.spec.coeffs)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    c_t, v_t = wl.make_insert_inputs_t(spec, dev)
    counts = c_t.cpu().numpy().view(np.uint32)
    values = v_t.cpu().numpy().view(np.uint32)
    N = values.shape[0]
    n_rand = max(1, w.n_random * rounds // 512)
    idx_r = wl.uniform_indices(w.read_seed, n_rand, N)
    idx_w = wl.uniform_indices(w.write_seed, n_rand, N)
    vals_w = wl.index_keyed_values(w.value_seed, idx_w, w.E)
    o = oracle.OracleGGArray(w.L, w.T, w.B, w.E)
    t = time.perf_counter()
    o.insert(counts, values)
    o.read(idx_r)
    o.write(idx_w, vals_w)
    o.sweep_add(1, 1)
    o.sweep_add(1, 1)
    o.flatten()
    dt = time.perf_counter() - t
    o.close()
    desc = (f"paper_growth 1024x512 B4096 int32 with {rounds} of 512 rounds ({N} elements), "
            f"{n_rand} random reads and writes, two +1 sweeps, flatten; single-threaded C++ oracle")
    return N, dt, desc


def cpu_baseline(rounds_full: int):
    rounds = max(1, min(rounds_full, 64))
    N, dt, desc = oracle_sample(rounds)
    return {"value": round(N / dt / 1e9, 5), "unit": "Gelem/s", "cores": 1, "kind": "oracle", "sample": desc,
            "seconds": round(dt, 3), "host_cores_available": os.cpu_count()}


def run_reference(args, world, rank):
    if rank != 0:
        return None
    # Size each step's sample so that warm-up + steps end within ~2 minutes.
    N1, dt1, _ = oracle_sample(4)
    per_round = dt1 / 4
    budget = 120.0 / max(1, args.steps + args.warmup)
    rounds = int(max(1, min(args.rounds, budget / max(per_round, 1e-6))))
    for _ in range(args.warmup):
        oracle_sample(rounds)
    tot_n, tot_t, desc = 0, 0.0, ""
    for _ in range(args.steps):
        n, dt, desc = oracle_sample(rounds)
        tot_n += n
        tot_t += dt
    value = tot_n / tot_t / 1e9
    return {
        "impl": "reference", "metric": METRIC, "value": round(value, 5), "unit": "Gelem/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(tot_t / args.steps * 1e3, 3),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
        "config": {"workload": f"paper_growth_1024x512_B4096_int32_R{args.rounds}", "sample_rounds": rounds},
        "cpu_baseline": {"value": round(value, 5), "unit": "Gelem/s", "cores": 1, "kind": "oracle",
                         "sample": desc},
        "e2e": {"value": round(value, 5), "unit": "Gelem/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }


def run_batched(args, world, rank, local):
    """4096 GGArrays of lognormal sizes (median 64K, sigma 1.5, capped 16M;
    int32/int64/16-byte records; Poisson(1) counts) grown to their targets:
    one captured clear+grow graph of the persistent batch kernel per step,
    against growing the same arrays with one launch sequence per array."""
    from paper_2209_00103_gb300 import batching
    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(dev)
    sizes = batching.batched_sizes(args.arrays)
    rule = batching.tuned_rule()
    pool, arrays, batch, params = batching.build(sizes, rule, stream)
    total = int(sizes.sum())
    bytes_written = int(sum(int(s) * batching.payload_bytes(a) for a, s in enumerate(sizes)))
    batch.capture(stream)
    for _ in range(max(3, args.warmup)):
        batch.replay(stream)
    torch.cuda.synchronize(dev)
    K = args.steps
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    sampler = ClockSampler(local)
    barrier(world)
    sampler.start()
    t0.record(stream)
    for _ in range(K):
        batch.replay(stream)
    t1.record(stream)
    torch.cuda.synchronize(dev)
    clocks = sampler.stop()
    ms = max_over_ranks(t0.elapsed_time(t1), world) / K
    value = sum_over_ranks(float(total), world) / (ms / 1e3) / 1e9
    ratio = batching.memory_ratio(arrays)
    plain_ms = batching.plain_time(arrays, sizes, stream)
    peak, _ = peaks()
    gbs = bytes_written / (ms / 1e3) / 1e9
    res = {"metric": f"batched GGArray growth Gelem/s ({len(sizes)} arrays, one persistent launch)", "value": round(value, 3),
           "unit": "Gelem/s", "n_gpus": world, "steps": K, "warmup": max(3, args.warmup),
           "ms_per_step": round(ms, 4), "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": "u32/u64/record", "data": "synthetic",
           "config": {"workload": f"batched_{len(sizes)}_lognormal_median64K_sigma1.5_cap16M", "arrays": len(sizes),
                      "elements": total, "bytes": bytes_written, "rule": rule.to_json() if hasattr(rule, "to_json") else rule.__dict__,
                      "step": "captured graph: clear every array + persistent grow kernels side by side + finalize"},
           "roofline": {"bound": "hbm", "achieved": round(gbs, 1), "peak": peak, "unit": "GB/s",
                        "frac": round(gbs / peak, 3), "traffic": None, "kernel": "batch_cluster_kernel + batch_grow_kernel (three payload sizes)",
                        "algorithmic_bytes_per_launch": bytes_written},
           "mem_over_needed": round(ratio, 4),
           "plain_one_launch_per_array": {"ms": round(plain_ms, 3),
                                          "gelem_s": round(total / (plain_ms / 1e3) / 1e9, 3),
                                          "speedup_of_batched": round(plain_ms / ms, 2)},
           # clear 2, a cluster and a block kernel per payload size, finalize
           "gpu_launches": K * 9, "clocks": clocks}
    batching.teardown(pool, arrays, batch)
    return res


def run_served(args, world, rank, local):
    """Poisson arrivals (20k req/s) over 65,536 live int64 arrays in a 64 GiB
    pool: 70% appends (n log-uniform 1..1M), 25% reads of 4096 random
    indices, 5% flattens that retire the array.  The same trace runs through
    the continuous-batching server and through the plain serial form (one
    request per launch sequence, each waited for)."""
    from paper_2209_00103_gb300 import serving
    cfg = serving.ServeConfig(duration=args.duration)
    if args.deadline is not None:
        cfg.deadline = args.deadline
    trace = serving.make_trace(cfg)
    srv = serving.Server(cfg)
    sampler = ClockSampler(local)
    sampler.start()
    rep = srv.run(trace, batched=True)
    clocks = sampler.stop()
    srv.close()
    plain = serving.Server(cfg)
    rep_plain = plain.run(trace, batched=False)
    plain.close()
    sweep = None if args.no_sweep else served_load_sweep(serving)
    return {"metric": "served GGArray p99 latency (ms), continuous batching", "value": rep["p99_ms"], "unit": "ms",
            "n_gpus": world, "steps": rep["completed"], "warmup": 0,
            "ms_per_step": round(rep["wall_s"] * 1e3 / max(1, rep["completed"]), 5), "higher_is_better": False,
            "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
            "config": {"workload": "served_65536_int64_arrays_poisson20k_70_25_5_pool64GiB",
                       "duration_s": cfg.duration, "requests": int(len(trace[0])), "arrays": cfg.n_arrays,
                       "L": cfg.L, "T": cfg.T, "B": cfg.B, "pool_bytes": cfg.pool_bytes,
                       "deadline_s": cfg.deadline, "max_inflight_steps": cfg.max_inflight},
            "served": rep, "plain_one_launch_per_request": rep_plain, "load_sweep": sweep, "clocks": clocks}


def set_l2_fetch_granularity(nbytes: int) -> int:
    """The current context's cudaLimitMaxL2FetchGranularity (a hint of this
    process's context, gone when it exits); returns the value in force."""
    import ctypes
    import glob
    lib = ctypes.CDLL(sorted(glob.glob(os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "lib64",
                                                    "libcudart.so*")))[-1])
    limit = 0x05   # cudaLimitMaxL2FetchGranularity
    if nbytes:
        assert lib.cudaDeviceSetLimit(limit, ctypes.c_size_t(nbytes)) == 0
    v = ctypes.c_size_t(0)
    assert lib.cudaDeviceGetLimit(ctypes.byref(v), limit) == 0
    return int(v.value)


def run_random_access(args, world, rank, local):
    """The step's random reads alone, beside a flat gather of the same
    indices: the paper-shaped array grown over --rounds rounds, 2^26 * R /
    512 uniform indices (the density of the full step), gga_read against
    torch.index_select on a flat copy.  For ncu captures of the two gathers
    (DRAM bytes per access) and of the L2 fetch-granularity hint."""
    from paper_2209_00103_gb300 import gga
    from paper_2209_00103_gb300 import workloads as wl
    dev = torch.device("cuda", local)
    gran = set_l2_fetch_granularity(args.l2_fetch)
    w = wl.paper_growth()
    R = args.rounds
    spec = wl.InsertSpec(L=w.L, T=w.T, E=w.E, seed=w.spec.seed, dist=w.spec.dist, rounds=R, coeffs=w.spec.coeffs)
    counts, values = wl.make_insert_inputs_t(spec, dev)
    N = int(values.shape[0])
    n_rand = max(1, w.n_random * R // 512)
    g = gga.GGArray(w.L, w.T, w.B, w.E, int(2.5 * N * w.E) + w.L * w.B * w.E * 4)
    stream = torch.cuda.current_stream(dev)
    g.insert(counts, values, stream)
    del counts
    idx = wl.uniform_indices_t(w.read_seed, n_rand, N, dev)
    out = gga.elem_tensor(n_rand, w.E, dev)
    del values
    flat = g.flatten()[:N]
    out_flat = torch.empty_like(out)

    def timed(fn, k=max(3, args.steps)):
        for _ in range(max(3, args.warmup)):
            fn()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(k)]
        for a, b in evs:
            a.record(stream)
            fn()
            b.record(stream)
        torch.cuda.synchronize(dev)
        return statistics.median(a.elapsed_time(b) for a, b in evs)

    ms_g = timed(lambda: g.read(idx, out, stream))
    ms_f = timed(lambda: torch.index_select(flat, 0, idx, out=out_flat))
    assert torch.equal(out, out_flat)
    g.close()
    peak, _ = peaks()
    alg = n_rand * (8 + 2 * w.E)
    return {"metric": "random reads G accesses/s (GGArray gga_read vs flat index_select)",
            "value": round(n_rand / (ms_g / 1e3) / 1e9, 3), "unit": "G accesses/s", "n_gpus": world,
            "steps": max(3, args.steps), "warmup": max(3, args.warmup), "ms_per_step": round(ms_g, 4),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
            "config": {"workload": f"paper_growth_1024x512_B4096_int32_R{R}_random_reads", "elements": N,
                       "reads": n_rand, "l2_fetch_granularity_bytes": gran},
            "gga_read": {"ms": round(ms_g, 4), "achieved_gbs": round(alg / (ms_g / 1e3) / 1e9, 1),
                         "frac_of_measured_peak": round(alg / (ms_g / 1e3) / 1e9 / peak, 3)},
            "flat_index_select": {"ms": round(ms_f, 4)}, "gpu_launches": 2 * max(3, args.steps)}


SWEEP_RATES = (20000.0, 50000.0, 100000.0, 200000.0, 500000.0, 1000000.0)
SWEEP_P99_BOUND_MS = 10.0


def served_load_sweep(serving, rates=SWEEP_RATES, p99_bound_ms=SWEEP_P99_BOUND_MS):
    """The same request mix at higher arrival rates, through both forms,
    over the window before the pool fills: each rate runs for half the time
    the offered appends (0.7 * rate * E[n] * 8 bytes per second, E[n] of the
    log-uniform sizes) take to fill the 64 GiB pool, at most 2 s.  A form
    sustains a rate when it completes every request with p99 latency at most
    p99_bound_ms and finishes within 10% of the trace's duration."""
    import math
    base = serving.ServeConfig()
    mean_n = (base.max_append - 1) / math.log(base.max_append)
    points = []
    for rate in rates:
        fill_s = base.pool_bytes / (base.mix[0] * rate * mean_n * base.E)
        cfg = serving.ServeConfig(rate=rate, duration=round(min(2.0, 0.5 * fill_s), 3))
        trace = serving.make_trace(cfg)
        point = {"rate_per_s": rate, "duration_s": cfg.duration, "requests": int(len(trace[0]))}
        for name, batched in (("batched", True), ("plain", False)):
            srv = serving.Server(cfg)
            r = srv.run(trace, batched=batched)
            srv.close()
            ok = (r["completed"] == r["requests"] and r.get("p99_ms", math.inf) <= p99_bound_ms
                  and r["wall_s"] <= 1.1 * cfg.duration)
            point[name] = {"p50_ms": r.get("p50_ms"), "p99_ms": r.get("p99_ms"), "elements_per_s": r["elements_per_s"],
                           "wall_s": r["wall_s"], "completed": r["completed"], "rejected": r["rejected"],
                           "requests_per_step": r["mean_requests_per_step"], "sustained": bool(ok)}
        points.append(point)
    best = {}
    for name in ("batched", "plain"):
        ok = [p for p in points if p[name]["sustained"]]
        best[name] = ({"rate_per_s": ok[-1]["rate_per_s"], "elements_per_s": ok[-1][name]["elements_per_s"]}
                      if ok else None)
    return {"p99_bound_ms": p99_bound_ms, "points": points, "highest_sustained": best}


def run_two_phase(args, world, rank, local):
    """The case study of the paper's Sec. VI-D: 2^24 initial 16-byte records
    over 1024 LFVectors x 512 threads, 8 generations of Geometric(1/2)-1
    children per record pushed back from inside the application kernel,
    then flatten and 20 streaming passes of pos += vel on the contiguous copy."""
    import numpy as np
    from paper_2209_00103_gb300 import gga
    from paper_2209_00103_gb300 import workloads as wl
    w = wl.two_phase(only_newborn=args.newborn, n0=args.n0, generations=args.generations)
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    counts = torch.from_numpy(wl.split_counts(w.L, w.T, w.n0).view(np.int32)).to(dev)
    recs = wl.initial_records_t(w.n0, dev)
    free, _ = torch.cuda.mem_get_info(dev)
    final_est = w.n0 * (w.generations + 1 if w.only_newborn else 2 ** w.generations)
    pool_bytes = int(min(2.3 * final_est * 16 + (1 << 30), free - final_est * 16 * 1.05 - (4 << 30)))
    g = gga.GGArray(w.L, w.T, w.B, 16, pool_bytes)
    born = torch.zeros(w.L, dtype=torch.int64, device=dev) if w.only_newborn else None
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(w.generations + 4)]
    offs = torch.zeros((w.generations + 1, w.L + 1), dtype=torch.int64, device=dev)
    ev[0].record(stream)
    g.insert(counts, recs, stream)
    ev[1].record(stream)
    gga.gga_offsets(g.h, offs[0], stream)
    for gen in range(w.generations):
        gga.gga_twophase_spawn(g.h, gen, w.seed, born, stream)
        ev[2 + gen].record(stream)
        gga.gga_offsets(g.h, offs[gen + 1], stream)   # sizes after the generation (8 KB copy, outside the events)
    n, rc = g.size(stream)
    if rc != gga.GGA_OK:
        raise RuntimeError(f"device error {rc}")
    mem = g.memory(stream)
    dst = gga.elem_tensor(n, 16, dev)
    a = torch.cuda.Event(enable_timing=True)
    b = torch.cuda.Event(enable_timing=True)
    c = torch.cuda.Event(enable_timing=True)
    a.record(stream)
    g.flatten(dst, stream)
    b.record(stream)
    gga.gga_twophase_work(dst, w.passes, stream)
    c.record(stream)
    torch.cuda.synchronize(dev)
    spawn_ms = ev[1].elapsed_time(ev[1 + w.generations])
    sizes = [int(x) for x in offs[:, w.L].cpu()]
    # Algorithmic bytes of the spawning: every parent record read (16 B), every child written (16 B).
    # All records spawn in reading A; in reading B only the previous generation's newborns do.
    spawn_bytes = 0
    for k in range(w.generations):
        parents = sizes[k] if not w.only_newborn else (sizes[k] - (sizes[k - 1] if k else 0))
        spawn_bytes += 16 * parents + 16 * (sizes[k + 1] - sizes[k])
    spawn_gen_ms = [ev[1 + k].elapsed_time(ev[2 + k]) for k in range(w.generations)]
    flat_ms = a.elapsed_time(b)
    work_ms = b.elapsed_time(c)
    peak, _ = peaks()
    spawned = n - w.n0
    res = {"metric": "two-phase case study: spawned records/s; flatten and work-pass GB/s",
           "value": round(spawned / (spawn_ms / 1e3) / 1e9, 3), "unit": "Grecords/s", "n_gpus": world,
           "steps": 1, "warmup": 0, "ms_per_step": round(ev[0].elapsed_time(ev[1 + w.generations]) + flat_ms + work_ms, 3),
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64/f32 records",
           "data": "synthetic",
           "config": {"workload": w.name, "initial_records": w.n0, "generations": w.generations,
                      "final_records": n, "spawning": "newborn" if w.only_newborn else "all records",
                      "passes": w.passes},
           "phases_ms": {"initial_insert": round(ev[0].elapsed_time(ev[1]), 3),
                         "spawn_generations": [round(x, 3) for x in spawn_gen_ms],
                         "flatten": round(flat_ms, 3), "work_passes": round(work_ms, 3)},
           "flatten_gbs": round(2 * n * 16 / (flat_ms / 1e3) / 1e9, 1),
           "flatten_frac_of_measured_peak": round(2 * n * 16 / (flat_ms / 1e3) / 1e9 / peak, 3),
           "work_pass_gbs_aos": round(w.passes * 32 * n / (work_ms / 1e3) / 1e9, 1),
           "records_after_generation": sizes,
           "spawn_gbs": round(spawn_bytes / (spawn_ms / 1e3) / 1e9, 1),
           "spawn_frac_of_measured_peak": round(spawn_bytes / (spawn_ms / 1e3) / 1e9 / peak, 3),
           "last_generation_gbs": round((16 * (sizes[-2] if not w.only_newborn else sizes[-2] - sizes[-3])
                                         + 16 * (sizes[-1] - sizes[-2])) / (spawn_gen_ms[-1] / 1e3) / 1e9, 1),
           "mem_over_needed": round(mem["bucket_bytes"] / max(1, mem["live_bytes"]), 4)}
    g.close()
    return res


def run_doubling(args, world, rank, local):
    """The growable-array experiment of the paper's Sec. VI-C (Table II):
    start at 10^6 int32 elements and double the size 10 times (to 1.024e9).
    Every doubling is a resize (capacity raised to twice the size: gga_reserve
    for a GGArray), an insertion of one element per element already there
    (gga_insert of one round: each LFVector's share split over its 1024
    threads, values packed in prefix-sum order), and a read/write pass adding
    +1 thirty times to every element (rw_b, the paper's per-block r/w).
    GGArray with 32 and 512 LFVectors (first bucket 4096), a static array
    allocated for the last size up front (no grow; contiguous copy for the
    insertion, +30 in one pass with PyTorch) and the memMap array (a reserved
    address range grown by mapping more physical memory, no copy)."""
    import numpy as np
    from paper_2209_00103_gb300 import gga
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    T, B, E = 1024, 4096, 4
    n0, iters = 1_000_000, 10
    final = n0 << iters
    values = torch.arange(final // 2, dtype=torch.int32, device=dev)     # the largest insertion's values

    def ev():
        return torch.cuda.Event(enable_timing=True)

    def split(n, parts):
        return np.array([n // parts + (1 if i < n % parts else 0) for i in range(parts)], dtype=np.int64)

    rows = {}
    for L in (32, 512):
        g = gga.GGArray(L, T, B, E, int(2.3 * final * E) + L * B * E * 4)
        sizes = np.zeros(L, dtype=np.int64)
        per_iter = []

        def insert_counts(add):
            c = np.zeros((1, L, T), dtype=np.uint32)
            for l in range(L):
                c[0, l, :] = split(int(add[l]), T)
            return torch.from_numpy(c.view(np.int32)).to(dev)

        # The initial 10^6 elements.
        add = split(n0, L)
        g.insert(insert_counts(add), values[:n0], stream)
        sizes += add
        for it in range(iters):
            target = torch.from_numpy((2 * sizes).astype(np.int64)).to(dev)
            counts = insert_counts(sizes)
            n_add = int(sizes.sum())
            torch.cuda.synchronize(dev)
            e = [ev() for _ in range(4)]
            e[0].record(stream)
            g.reserve(target, stream)
            e[1].record(stream)
            g.insert(counts, values[:n_add], stream)
            e[2].record(stream)
            g.sweep(gga.GGA_RW_B, 1, 30, stream)
            e[3].record(stream)
            torch.cuda.synchronize(dev)
            sizes = 2 * sizes
            per_iter.append({"size_after": int(sizes.sum()), "grow_ms": round(e[0].elapsed_time(e[1]), 4),
                             "insert_ms": round(e[1].elapsed_time(e[2]), 4), "rw_ms": round(e[2].elapsed_time(e[3]), 4)})
        n, rc = g.size(stream)
        if rc != gga.GGA_OK or n != final:
            raise RuntimeError(f"doubling GGArray{L}: size {n} vs {final}, device error {rc}")
        mem = g.memory(stream)
        rows[f"GGArray{L}"] = {"last": per_iter[-1], "iterations": per_iter,
                               "mem_over_needed": round(mem["bucket_bytes"] / max(1, mem["live_bytes"]), 4)}
        g.close()

    # Static: allocated for the last size; insertion is a contiguous copy after the size.
    a = torch.zeros(final, dtype=torch.int32, device=dev)
    size = n0
    a[:n0].copy_(values[:n0])
    per_iter = []
    for it in range(iters):
        torch.cuda.synchronize(dev)
        e = [ev() for _ in range(3)]
        e[0].record(stream)
        a[size:2 * size].copy_(values[:size])
        e[1].record(stream)
        a[:2 * size].add_(30)
        e[2].record(stream)
        torch.cuda.synchronize(dev)
        size *= 2
        per_iter.append({"size_after": size, "grow_ms": None, "insert_ms": round(e[0].elapsed_time(e[1]), 4),
                         "rw_ms": round(e[1].elapsed_time(e[2]), 4)})
    rows["static"] = {"last": per_iter[-1], "iterations": per_iter, "mem_over_needed": 1.0}
    del a

    # memMap: a reserved address range grown by mapping physical memory (no copy);
    # grow is the host's mapping calls (wall clock), then the same insert and r/w.
    vm = gga.GGAVMM(final * E)
    size = n0
    vm.grow(size * E)
    vm.tensor(size)[:].copy_(values[:n0])
    per_iter = []
    for it in range(iters):
        torch.cuda.synchronize(dev)
        t_g = time.perf_counter()
        vm.grow(2 * size * E)
        grow_ms = (time.perf_counter() - t_g) * 1e3
        view = vm.tensor(2 * size)
        e = [ev() for _ in range(3)]
        e[0].record(stream)
        view[size:2 * size].copy_(values[:size])
        e[1].record(stream)
        view.add_(30)
        e[2].record(stream)
        torch.cuda.synchronize(dev)
        size *= 2
        per_iter.append({"size_after": size, "grow_ms": round(grow_ms, 4), "insert_ms": round(e[0].elapsed_time(e[1]), 4),
                         "rw_ms": round(e[1].elapsed_time(e[2]), 4)})
        del view
    rows["memMap"] = {"last": per_iter[-1], "iterations": per_iter,
                      "mem_over_needed": round(vm.info()["mapped_bytes"] / (final * E), 4),
                      "grow": "host calls mapping the new physical memory (wall clock)"}
    torch.cuda.synchronize(dev)
    vm.close()

    last512 = rows["GGArray512"]["last"]
    peak, _ = peaks()
    ins_bytes = (final // 2) * 2 * E + 512 * T * 4          # values read + elements written + counts
    rw_bytes = final * 2 * E
    return {"metric": "growable-array doubling (Sec. VI-C, Table II): last doubling 5.12e8 -> 1.024e9 int32",
            "value": round((final // 2) / (last512["insert_ms"] / 1e3) / 1e9, 3), "unit": "Gelem/s (GGArray512 insert)",
            "n_gpus": world, "steps": iters, "warmup": 0, "ms_per_step": round(
                last512["grow_ms"] + last512["insert_ms"] + last512["rw_ms"], 4),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
            "config": {"workload": "doubling_1e6_x2_10_int32", "T": T, "B": B, "start": n0, "final": final},
            "roofline": {"bound": "hbm", "kernel": "GGArray512 insertion (count + tile scan + reserve + copy)",
                         "achieved": round(ins_bytes / (last512["insert_ms"] / 1e3) / 1e9, 1), "peak": peak,
                         "unit": "GB/s", "frac": round(ins_bytes / (last512["insert_ms"] / 1e3) / 1e9 / peak, 3),
                         "traffic": None},
            "rw_gbs_GGArray512": round(rw_bytes / (last512["rw_ms"] / 1e3) / 1e9, 1),
            "table": rows,
            "paper_table_ii_a100_ms": {"static": {"grow": None, "insert": 7.07, "rw": 6.27},
                                       "memMap": {"grow": 5.21, "insert": 7.87, "rw": 6.28},
                                       "GGArray512": {"grow": 8.76, "insert": 11.79, "rw": 69.73},
                                       "GGArray32": {"grow": 0.52, "insert": 27.90, "rw": 198.32}}}


def run_insertion(args, world, rank, local):
    """The insertion experiment of the paper's Sec. VI-A: a static (flat)
    array of 10^6 int32 elements with room to double 10 times; each doubling
    inserts one element per element already there, with one thread per new
    element, by Sec. III-B's atomic approach (one atomicAdd per thread) and by
    its warp-shuffle scan approach (one atomicAdd per block), for several
    block sizes.  (The tensor-core scan is not built.)"""
    from paper_2209_00103_gb300 import gga
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    n0, iters = 1_000_000, 10
    final = n0 << iters
    a = torch.empty(final, dtype=torch.int32, device=dev)
    size = torch.zeros(1, dtype=torch.int64, device=dev)
    rows = {}
    for mode, name in ((gga.GGA_FLAT_SCAN, "scan"), (gga.GGA_FLAT_ATOMIC, "atomic")):
        for T in (128, 256, 512, 1024):
            size.fill_(n0)
            s_host = n0
            per_iter = []
            for it in range(iters):
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                gga.gga_flat_insert(mode, a, size, s_host, T, s_host, stream)
                e1.record(stream)
                torch.cuda.synchronize(dev)
                s_host *= 2
                per_iter.append(round(e0.elapsed_time(e1), 4))
            if int(size.item()) != final:
                raise RuntimeError(f"insertion {name} T={T}: size {int(size.item())} vs {final}")
            rows[f"{name}_T{T}"] = {"iterations_ms": per_iter, "last_ms": per_iter[-1],
                                    "last_gelem_s": round((final // 2) / (per_iter[-1] / 1e3) / 1e9, 2)}
    best_scan = min((v["last_ms"], k) for k, v in rows.items() if k.startswith("scan"))
    best_atomic = min((v["last_ms"], k) for k, v in rows.items() if k.startswith("atomic"))
    peak, _ = peaks()
    gbs = (final // 2) * 4 / (best_scan[0] / 1e3) / 1e9
    return {"metric": "insertion approaches on a flat array (Sec. VI-A): last doubling 5.12e8 -> 1.024e9 int32",
            "value": round((final // 2) / (best_scan[0] / 1e3) / 1e9, 3), "unit": "Gelem/s (best scan)",
            "n_gpus": world, "steps": iters, "warmup": 0, "ms_per_step": best_scan[0], "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
            "config": {"workload": "flat_insertion_doubling_1e6_x2_10_int32", "start": n0, "final": final},
            "roofline": {"bound": "hbm", "kernel": f"flat_insert_scan_kernel ({best_scan[1]})", "achieved": round(gbs, 1),
                         "peak": peak, "unit": "GB/s", "frac": round(gbs / peak, 3), "traffic": None},
            "best": {"scan": best_scan[1], "atomic": best_atomic[1],
                     "atomic_over_scan": round(best_atomic[0] / best_scan[0], 2)},
            "table": rows}


def run_phases(args, world, rank, local):
    """The two-phase case study of the paper's Sec. VI-D, against memMap:
    every iteration inserts k times the array's size (k = 1, 3, 10), then
    runs a work phase of W kernels adding 1 to every element (W = 1 .. 1000);
    four iterations, starting from 10^9 / (1+k)^4 so that the final size is
    10^9 int32.  GGArray (512 LFVectors, 1024 threads, first bucket 4096):
    insertion with gga_insert, then flatten into a contiguous array the work
    runs on.  memMap: grow by mapping, the insertion copied into the mapped
    range, the work on it directly.  Host wall time of all iterations,
    synchronized before and after; speedup = memMap time / GGArray time."""
    import numpy as np
    from paper_2209_00103_gb300 import gga
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    L, T, B, E, iters = 512, 1024, 4096, 4, 4
    Ws = (1, 10, 100, 1000)
    final_target = 10 ** 9

    def split(n, parts):
        return np.array([n // parts + (1 if i < n % parts else 0) for i in range(parts)], dtype=np.int64)

    # Warm-up: load every kernel both variants use (insert, flatten, the +1
    # pass, the mapping calls) before anything is timed.
    wg = gga.GGArray(L, T, B, E, 64 << 20)
    wc = torch.ones((1, L, T), dtype=torch.int32, device=dev)
    wv = torch.arange(L * T, dtype=torch.int32, device=dev)
    wg.insert(wc, wv, stream)
    wf = torch.empty(L * T, dtype=torch.int32, device=dev)
    wg.flatten(wf, stream)
    wf.add_(1)
    wvm = gga.GGAVMM(64 << 20)
    wvm.grow(4 << 20)
    wvm.tensor(1 << 20)[:].copy_(wv[:1 << 19].repeat(2))
    wvm.tensor(1 << 20).add_(1)
    torch.cuda.synchronize(dev)
    wvm.close()
    wg.close()
    del wc, wv, wf

    out = {}
    for k in (1, 3, 10):
        start = round(final_target / (1 + k) ** iters)
        final = start * (1 + k) ** iters
        max_add = final - final // (1 + k)
        values = torch.arange(max_add, dtype=torch.int32, device=dev)
        flat = torch.empty(final, dtype=torch.int32, device=dev)
        rows = {}
        for W in Ws:
            # GGArray
            g = gga.GGArray(L, T, B, E, int(2.3 * final * E) + L * B * E * 4)
            sizes = split(start, L)
            c0 = np.zeros((1, L, T), dtype=np.uint32)
            for l in range(L):
                c0[0, l, :] = split(int(sizes[l]), T)
            g.insert(torch.from_numpy(c0.view(np.int32)).to(dev), values[:start], stream)
            counts = []
            sz = sizes.copy()
            for it in range(iters):
                c = np.zeros((1, L, T), dtype=np.uint32)
                for l in range(L):
                    c[0, l, :] = split(int(k * sz[l]), T)
                counts.append(torch.from_numpy(c.view(np.int32)).to(dev))
                sz = sz * (1 + k)
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            n = start
            t_ins = t_flat = 0.0
            for it in range(iters):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
                e[0].record(stream)
                g.insert(counts[it], values[:k * n], stream)
                e[1].record(stream)
                n = n * (1 + k)
                g.flatten(flat[:n], stream)
                e[2].record(stream)
                view = flat[:n]
                for _ in range(W):
                    view.add_(1)
                torch.cuda.synchronize(dev)
                t_ins += e[0].elapsed_time(e[1])
                t_flat += e[1].elapsed_time(e[2])
            gg_ms = (time.perf_counter() - t0) * 1e3
            if g.size(stream)[0] != final:
                raise RuntimeError("phases: GGArray size mismatch")
            g.close()
            # memMap
            vm = gga.GGAVMM(final * E)
            vm.grow(start * E)
            vm.tensor(start)[:].copy_(values[:start])
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            n = start
            for it in range(iters):
                vm.grow((1 + k) * n * E)
                view = vm.tensor((1 + k) * n)
                view[n:].copy_(values[:k * n])
                n = n * (1 + k)
                for _ in range(W):
                    view.add_(1)
                del view
            torch.cuda.synchronize(dev)
            mm_ms = (time.perf_counter() - t0) * 1e3
            vm.close()
            rows[f"W{W}"] = {"ggarray_ms": round(gg_ms, 3), "ggarray_insert_ms": round(t_ins, 3),
                             "ggarray_flatten_ms": round(t_flat, 3), "memmap_ms": round(mm_ms, 3),
                             "speedup_ggarray_over_memmap": round(mm_ms / gg_ms, 3)}
        out[f"k{k}"] = {"start": start, "final": final, "rows": rows}
        del values, flat
    w1 = out["k1"]["rows"]["W1"]
    return {"metric": "two-phase case study (Sec. VI-D): speedup of GGArray over memMap",
            "value": w1["speedup_ggarray_over_memmap"], "unit": "x (k=1, W=1)", "n_gpus": world,
            "steps": iters, "warmup": 0, "ms_per_step": w1["ggarray_ms"], "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
            "config": {"workload": "two_phase_vs_memmap_final1e9_int32", "L": L, "T": T, "B": B,
                       "iterations": iters, "insert_factors": [1, 3, 10], "work_kernels": list(Ws)},
            "table": out}


def main():
    args = parse_args()
    world, rank, local = dist_setup()
    if args.impl == "reference":
        res = run_reference(args, world, rank)
    elif args.workload == "batched":
        res = run_batched(args, world, rank, local)
    elif args.workload == "served":
        res = run_served(args, world, rank, local)
    elif args.workload == "two_phase":
        res = run_two_phase(args, world, rank, local)
    elif args.workload == "doubling":
        res = run_doubling(args, world, rank, local)
    elif args.workload == "insertion":
        res = run_insertion(args, world, rank, local)
    elif args.workload == "phases":
        res = run_phases(args, world, rank, local)
    elif args.workload == "random_access":
        res = run_random_access(args, world, rank, local)
    else:
        res = run_ours(args, world, rank, local)
    if rank == 0 and res is not None:
        print(json.dumps(res), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
