#!/usr/bin/env python
"""Benchmark of the short-range P3M hot path on GB300.

One step = one pass of the whole forward hot path over the 128^3 clustered
particle set (30% uniform + 70% in 4096 Plummer spheres, PM grid 256^3,
x_s = 1.25/256, x_r = 4.5 x_s, B-spline softening), all particles active:

  sort into tiles/subtiles (momenta and rungs carried) -> receiver work list
  -> FP32 short-range accelerations -> rung assignment -> kick -> drift

Reported value: interacting ordered pairs (i active, j != i, r < x_r) per
second of device time.  Also reported: the FP64 path's rate, the adjoint
(VJP) kernel time over the forward kernel time, the pair kernel's fraction of
the FP32 ALU roofline, an end-to-end figure through host buffers, and the CPU
oracle on a bounded sample of receivers.

Usage:  python bench.py [--gpus N --steps K --warmup W] [--impl reference]
For N > 1 launch with torch.distributed.run; ranks run independent replicas
(distinct seeds) and the value is the sum over ranks divided by the slowest
rank's time (weak scaling).
"""
from __future__ import annotations

import argparse
import hashlib
import re
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "short-range pair-interactions/s (FP32 vs FP64 path) at ≤1e-5 rel RMS force; adjoint time/fwd"
UNIT = "pair-interactions/s"
SM_COUNT = 152
FP32_LANES_PER_SM = 128
SM_MAX_MHZ = 2070.0
OPS_PER_PAIR = 26  # FP32 pipe instructions per interacting pair, one-sided (gathering) kernel
OPS_PER_PAIR_SYM = 29  # per unordered pair in the Newton-III kernel: the same 26 + 3 for the partner's sum


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--mode", choices=["replicas", "slabs"], default="replicas",
                    help="N > 1: independent replicas (weak scaling) or the slab decomposition of one set "
                         "with halo exchange (strong scaling)")
    ap.add_argument("--workload", default="n2m")
    ap.add_argument("--cpu-sample", type=int, default=1 << 18, help="receivers in the CPU-oracle sample")
    ap.add_argument("--ref-sample", type=int, default=1 << 14, help="receivers per reference-arm step")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--evolve", type=int, default=0,
                    help="profiling modes: benchmark steps applied to the set before the measurement")
    ap.add_argument("--no-large", action="store_true",
                    help="skip the 512^3 and 1024^3 sub-records (full step, rung substeps, FP32 vs FP64)")
    ap.add_argument("--only", choices=["forces32", "forces32_gather", "forces64", "vjp32", "sort", "pm32",
                                       "rung_steps", "kick", "substep"],
                    default=None,
                    help="profiling mode: run just one kernel family (no contract line)")
    return ap.parse_args()


def source_hash(paths):
    """Hash of the kernel sources' code: comments dropped and whitespace runs collapsed,
    so that a change of wording alone does not retire a profile."""
    h = hashlib.sha256()
    for p in paths:
        with open(os.path.join(ROOT, p), encoding="utf-8") as f:
            text = f.read()
        text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
        text = re.sub(r"//[^\n]*", " ", text)
        h.update(" ".join(text.split()).encode())
    return h.hexdigest()[:16]


HBM_FALLBACK_GBS = 6800.0  # the profiling recipe's fallback, used only without MEASURED_PEAKS.json
SORT_BYTES_PER_PARTICLE = 110  # read/write x, ids, perm, carried momenta and rungs (algorithmic)
KICK_DRIFT_BYTES_PER_PARTICLE = 109  # read a (FP32) 12, r/w q 48, r/w x 48, write rung 1


def hbm_peak():
    """Measured copy bandwidth of this GPU (GB/s) and where it came from."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            return float(json.load(f)["hbm_gbs"]), "measured"
    except Exception:
        return HBM_FALLBACK_GBS, "fallback"


FORCE_SOURCES = ["paper_2112_01508_gb300/csrc/force.cu", "paper_2112_01508_gb300/csrc/pair_math.cuh",
                 "paper_2112_01508_gb300/csrc/traverse.cuh", "paper_2112_01508_gb300/csrc/common.cuh"]


class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi while running."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.file = None

    def start(self):
        try:
            self.file = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=self.file, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.file.flush()
        rows = []
        with open(self.file.name) as f:
            for line in f:
                parts = [x.strip() for x in line.split(",")]
                if len(parts) >= 8:
                    rows.append(parts)
        os.unlink(self.file.name)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = [float(r[0]) for r in rows if r[0].replace(".", "").isdigit()]
        mx = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in rows for k in range(4) if r[4 + k].lower() == "active"})
        power = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        loaded = [s for s in sm if s > 0.5 * (max(mx) if mx else 1)] or sm
        return {"sm_mhz": statistics.median(loaded) if loaded else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons, "samples": len(rows),
                "power_w_max": max(power) if power else None}


def dist_setup():
    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    elif torch.cuda.is_available():
        torch.cuda.set_device(local)
    return world, rank, local


def _reduce(value: float, world: int, op_name: str) -> float:
    """All-reduce one scalar over the ranks (NCCL on GPUs, gloo on CPU)."""
    if world == 1:
        return value
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([value], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=getattr(dist.ReduceOp, op_name))
    return float(t.item())


def max_over_ranks(value: float, world: int) -> float:
    return _reduce(value, world, "MAX")


def sum_over_ranks(value: float, world: int) -> float:
    return _reduce(value, world, "SUM")


def barrier(world: int):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def cpu_oracle_rate(w, pos, n_recv: int, seed: int = 7):
    """The CPU oracle as it stands, on a bounded sample of receivers (all suppliers)."""
    import numpy as np

    import oracle
    rng = np.random.default_rng(seed)
    recv = np.sort(rng.choice(w.n, size=min(n_recv, w.n), replace=False))
    t0 = time.perf_counter()
    _, pairs = oracle.sr_accel_subset(pos, recv, w.x_s, w.x_r, w.G_m, "bspline", w.eps)
    dt = time.perf_counter() - t0
    return float(pairs.sum()) / dt, dt, int(pairs.sum()), len(recv), oracle.num_threads()


def traffic_from_profiles(workload: str):
    """DRAM traffic of the pair kernel from the committed ncu summary, if it was
    captured on this workload and the current kernel source (else None)."""
    p = os.path.join(ROOT, "profiles", f"force_f32_{workload}.json")
    if not os.path.exists(p):
        return None
    try:
        with open(p) as f:
            d = json.load(f)
        if d.get("source_hash") != source_hash(FORCE_SOURCES):
            return None
        return d.get("dram_bytes_per_launch")
    except Exception:
        return None


def large_record(wname: str, dev, with_cpu: bool, steps: int = 2):
    """Sub-record for a large workload (512^3: 8 rungs, per-rung substeps; 1024^3: full
    step and deepest-rung substep, FP32 vs FP64).  The CPU-baseline leg runs the oracle
    on 2^18 seeded receivers of the same state (all suppliers); the GPU outputs on those
    receivers are compared with it."""
    import numpy as np
    import torch

    import synth
    from paper_2112_01508_gb300 import ShortRange

    w = synth.workload(wname)
    n = w.n
    eta, n_rung = 0.025, 8
    t0 = time.perf_counter()
    pos_np = synth.workload_positions(w)
    rec = {"workload": f"{w.name}: {w.description}", "n": n, "n_sub": w.n_sub, "softening": "bspline",
           "generate_s": time.perf_counter() - t0}
    stream = torch.cuda.current_stream(dev)
    gen = torch.Generator(device=dev)
    with ShortRange.from_workload(w, device=dev) as sr:
        p = torch.from_numpy(pos_np).to(dev)
        perm = torch.empty(n, dtype=torch.int32, device=dev)
        sr.sort(p, perm_out=perm)
        sr.build_pairs()
        a32 = sr.forces(p, 32)
        ts = []
        for _ in range(2):
            sr.forces(p, 32, a32)
            ts.append(sr.stats().force_kernel_ms)
        st = sr.stats()
        peak = SM_COUNT * FP32_LANES_PER_SM * SM_MAX_MHZ * 1e6 / OPS_PER_PAIR
        rec["full_fp32"] = {"pairs": st.pairs_last, "kernel_ms": statistics.mean(ts),
                            "value": st.pairs_last / (statistics.mean(ts) * 1e-3), "unit": UNIT,
                            "kernel": "k_force_sym<bspline> (each pair once)",
                            "frac": st.pairs_last / (statistics.mean(ts) * 1e-3) / peak}
        # rungs from the fake kick (Eq. rung), dt putting ~1% of the particles on rung 7
        amag = torch.linalg.vector_norm(a32, dim=0)
        gen.manual_seed(0)
        q99 = float(torch.quantile(amag[torch.randperm(n, device=dev, generator=gen)[:1 << 20]], 0.99))
        del amag
        dt = 64.0 * (2.0 * eta * w.eps / q99) ** 0.5
        rung = sr.assign_rungs(a32, dt, eta, w.eps)
        rec["rung_histogram"] = torch.bincount(rung.long(), minlength=n_rung).tolist()
        rng = np.random.default_rng(11)
        k32 = np.sort(rng.choice(n, size=1 << 18, replace=False))
        g32 = a32[:, torch.from_numpy(k32).to(dev)].double().cpu().numpy()
        subs = {}
        for lc in range(n_rung):
            sr.build_pairs(None if lc == 0 else rung, lc)
            sr.forces(p, 32, a32)
            st = sr.stats()
            subs[str(lc)] = {"receivers": st.n_active, "pairs": st.pairs_last,
                             "force_kernel_ms": st.force_kernel_ms,
                             "kernel_frac": st.pairs_last / (st.force_kernel_ms * 1e-3) / peak}
        rec["rung_substeps"] = subs
        # deepest-rung substep, FP32 and FP64 (receivers: rung 7; suppliers: all)
        sr.build_pairs(rung, n_rung - 1)
        sr.forces(p, 32, a32)
        st32 = sr.stats()
        a64 = torch.full((3, n), float("nan"), dtype=torch.float64, device=dev)
        sr.forces(p, 64, a64)
        st64 = sr.stats()
        act = torch.nonzero(rung >= n_rung - 1).flatten()
        gen.manual_seed(1)
        k64 = torch.sort(act[torch.randperm(len(act), device=dev, generator=gen)[:1 << 18]]).values
        g64 = a64[:, k64].cpu().numpy()
        k64 = k64.cpu().numpy()
        del a64
        rec["deepest_rung"] = {
            "rung": n_rung - 1, "receivers": st32.n_active, "pairs": st32.pairs_last,
            "fp32_kernel_ms": st32.force_kernel_ms, "fp64_kernel_ms": st64.force_kernel_ms,
            "fp32_value": st32.pairs_last / (st32.force_kernel_ms * 1e-3),
            "fp64_value": st64.pairs_last / (st64.force_kernel_ms * 1e-3),
            "fp32_over_fp64": st64.force_kernel_ms / st32.force_kernel_ms, "unit": UNIT}
        perm_np = perm.cpu().numpy().astype(np.int64)
        # the full step (sort with momenta and rungs carried, work list, FP32 forces,
        # rungs + kick + drift), all particles receivers; FP32 momenta at 1024^3
        mom = torch.zeros((3, n), dtype=torch.float32 if n > (1 << 28) else torch.float64, device=dev)
        kick_factor = [dt / 2 ** l for l in range(n_rung)]
        step_ms, step_pairs = [], []
        scr = [torch.empty_like(p), torch.empty_like(mom), torch.empty_like(rung)]
        for k in range(1 + steps):
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            sr.sort(p, carry=[mom, rung], scratch=scr)
            sr.build_pairs()
            sr.forces(p, 32, a32)
            sr.kick_drift(p, mom, a32, rung, dt, eta, w.eps, kick_factor, dt / 2 ** (n_rung - 1))
            e1.record(stream)
            st = sr.stats()
            if k > 0:
                step_ms.append(e0.elapsed_time(e1))
                step_pairs.append(st.pairs_last)
        rec["full_step"] = {"ms": statistics.mean(step_ms), "pairs": statistics.mean(step_pairs),
                            "value": sum(step_pairs) / (sum(step_ms) * 1e-3), "unit": UNIT,
                            "momenta": str(mom.dtype).replace("torch.", ""),
                            "step": "sort+carry, work list, FP32 forces, rungs+kick+drift"}
        del p, a32, mom, rung, scr
    torch.cuda.empty_cache()
    if with_cpu:
        import oracle
        t0 = time.perf_counter()
        ref32, pc = oracle.sr_accel_subset(pos_np, perm_np[k32], w.x_s, w.x_r, w.G_m, "bspline", w.eps)
        secs = time.perf_counter() - t0
        ref64, _ = oracle.sr_accel_subset(pos_np, perm_np[k64], w.x_s, w.x_r, w.G_m, "bspline", w.eps)

        def rel(a, b):
            return float(np.sqrt(((a - b) ** 2).sum() / (b ** 2).sum()))
        rec["cpu_baseline"] = {"value": float(pc.sum()) / secs, "unit": UNIT, "cores": oracle.num_threads(),
                               "kind": "oracle",
                               "sample": f"{len(k32)} seeded receivers of the initial state (all {n} suppliers; "
                                         f"includes the cell-list build), {int(pc.sum())} pairs, {secs:.1f} s"}
        rec["parity"] = {"receivers": len(k32), "fp32_all_active_rel_rms": rel(g32, ref32),
                         "fp64_deepest_rung_rel_rms": rel(g64, ref64), "tolerance": {"fp32": 1e-5, "fp64": 1e-12}}
    return rec


def run_ours(args):
    import numpy as np
    import torch

    import synth
    from paper_2112_01508_gb300 import ShortRange

    world, rank, local = dist_setup()
    dev = torch.device("cuda", local)
    w = synth.workload(args.workload)
    n = w.n
    seed = w.seed + 1000 * rank  # independent replica per rank
    pos_np = synth.positions(n, seed, w.frac_uniform, w.n_spheres, w.b_lo, w.b_hi)
    pos_host = torch.from_numpy(pos_np).pin_memory()
    mom_host = torch.zeros((3, n), dtype=torch.float64).pin_memory()
    acc_host = torch.empty((3, n), dtype=torch.float32).pin_memory()
    pos = pos_host.to(dev)
    pos0 = pos.clone()
    mom = torch.zeros((3, n), dtype=torch.float64, device=dev)
    rung = torch.zeros(n, dtype=torch.int8, device=dev)
    acc = torch.zeros((3, n), dtype=torch.float32, device=dev)
    acc64 = torch.zeros((3, n), dtype=torch.float64, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)  # > 129 MB L2
    sr = ShortRange.from_workload(w, device=dev)
    eta, n_rung = 0.025, 8

    # time step from the fake kick (Section 2.2.2): 1% of particles on the top rung
    sr.sort(pos)
    sr.build_pairs()
    sr.forces(pos, 64, acc64)
    amag = torch.linalg.vector_norm(acc64, dim=0)
    q99 = float(torch.quantile(amag[torch.randperm(n, device=dev)[:1 << 20]].float(), 0.99))
    dt = 64.0 * (2.0 * eta * w.eps / max(q99, 1e-30)) ** 0.5
    kick_factor = [dt / 2 ** l for l in range(n_rung)]
    drift_factor = dt / 2 ** (n_rung - 1)

    def step(ev=None):
        if ev is not None:
            ev[0].record(stream)
        sr.sort(pos, carry=[mom, rung], scratch=scratch)  # out of place, storages swapped
        if ev is not None:
            ev[1].record(stream)
        sr.build_pairs()
        sr.forces(pos, 32, acc)
        if ev is not None:
            ev[2].record(stream)
        sr.kick_drift(pos, mom, acc, rung, dt, eta, w.eps, kick_factor, drift_factor)
        if ev is not None:
            ev[3].record(stream)

    stream = torch.cuda.current_stream(dev)
    scratch = [torch.empty_like(pos), torch.empty_like(mom), torch.empty_like(rung)]
    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()

    vis = [v for v in os.environ.get("CUDA_VISIBLE_DEVICES", "").split(",") if v.strip().isdigit()]
    sampler = ClockSampler(int(vis[local]) if local < len(vis) else local)
    launches0 = sr.stats().kernel_launches
    step_ms, kern_ms, pairs, sort_ms, kd_ms = [], [], [], [], []
    barrier(world)
    torch.cuda.synchronize()
    sampler.start()
    torch.cuda.nvtx.range_push("timed")
    t_wall0 = time.perf_counter()
    for _ in range(args.steps):
        flush.zero_()
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
        step(ev)
        st = sr.stats()  # synchronises the stream
        step_ms.append(ev[0].elapsed_time(ev[3]))
        sort_ms.append(ev[0].elapsed_time(ev[1]))
        kd_ms.append(ev[2].elapsed_time(ev[3]))
        kern_ms.append(st.force_kernel_ms)
        pairs.append(st.pairs_last)
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_pop()
    barrier(world)
    t_wall = time.perf_counter() - t_wall0
    clocks = sampler.stop()
    launches = sr.stats().kernel_launches - launches0

    total_ms_local = sum(step_ms)
    total_ms = max_over_ranks(total_ms_local, world)
    total_pairs = sum_over_ranks(float(sum(pairs)), world)
    value = total_pairs / (total_ms * 1e-3)
    ms_per_step = total_ms / args.steps

    # dominant kernel: the FP32 pair kernel, timed live with events around its launch
    kern_avg_ms = statistics.mean(kern_ms)
    pairs_avg = statistics.mean(pairs)
    achieved = pairs_avg / (kern_avg_ms * 1e-3)
    lane_rate = SM_COUNT * FP32_LANES_PER_SM * SM_MAX_MHZ * 1e6
    # the unit of work is the ordered interacting pair at its fixed algorithmic cost of 26 FP32
    # instructions; the all-active step runs the each-pair-once kernel, whose evaluations serve
    # two ordered interactions each (its own minimum, 29 per unordered pair, is reported beside)
    peak = lane_rate / OPS_PER_PAIR
    roofline = {"bound": "alu", "achieved": achieved / 1e9, "peak": peak / 1e9, "unit": "Gpair/s",
                "frac": achieved / peak, "traffic": traffic_from_profiles(w.name),
                "kernel": "k_force_sym<bspline> (FP32 forward, each pair once)", "kernel_ms": kern_avg_ms,
                "peak_basis": f"{SM_COUNT} SMs x {FP32_LANES_PER_SM} FP32 lanes x {SM_MAX_MHZ:.0f} MHz / "
                              f"{OPS_PER_PAIR} FP32 ops per interacting pair",
                "frac_of_each_pair_once_minimum": achieved / (2.0 * lane_rate / OPS_PER_PAIR_SYM)}

    # HBM-bound phases of the step against the measured copy bandwidth
    peak_gbs, peak_src = hbm_peak()

    def hbm_rec(bytes_per_particle, ms_list, what):
        ms = statistics.mean(ms_list)
        gbs = bytes_per_particle * n / (ms * 1e-3) / 1e9
        return {"what": what, "bytes_per_step": bytes_per_particle * n, "ms": ms, "gbs": gbs,
                "frac": gbs / peak_gbs}
    hbm = {"peak_gbs": peak_gbs, "peak_source": peak_src,
           "sort": hbm_rec(SORT_BYTES_PER_PARTICLE, sort_ms,
                           "p3m_sr_sort: bin, subtile offsets, stable radix sort, gathers of positions, "
                           "momenta and rungs, FP32 records (algorithmic 110 B per particle)"),
           "kick": hbm_rec(KICK_DRIFT_BYTES_PER_PARTICLE, kd_ms,
                           "p3m_sr_kick_drift: Eq. rung, kick and drift in one pass (algorithmic 109 B per "
                           "particle)")}

    # FP64 path and adjoint on the same (current) particle state
    sr.sort(pos, carry=[mom, rung])
    sr.build_pairs()
    fp64_ms = []
    for _ in range(3):
        flush.zero_()
        sr.forces(pos, 64, acc64)
        fp64_ms.append(sr.stats().force_kernel_ms)
    fp64_pairs = sr.stats().pairs_last
    fwd_ms, vjp_ms = [], []
    abar = torch.randn((3, n), dtype=torch.float32, device=dev)
    for _ in range(3):
        flush.zero_()
        sr.forces(pos, 32, acc)
        fwd_ms.append(sr.stats().force_kernel_ms)
        flush.zero_()
        sr.vjp(pos, abar, 32)
        vjp_ms.append(sr.stats().vjp_kernel_ms)
    a32 = acc.double()
    parity_32_64 = float(torch.sqrt(((a32 - acc64) ** 2).sum() / (acc64 ** 2).sum()))
    # the one-sided (gathering) FP32 kernel on the same state: each pair from both sides
    sr.set_symmetric(False)
    gat_ms = []
    acc_g = torch.zeros_like(acc)
    for _ in range(3):
        flush.zero_()
        sr.forces(pos, 32, acc_g)
        gat_ms.append(sr.stats().force_kernel_ms)
    sr.set_symmetric(True)
    gat_rate = sr.stats().pairs_last / (statistics.mean(gat_ms) * 1e-3)
    one_sided = {"value": gat_rate, "unit": UNIT, "kernel_ms": statistics.mean(gat_ms),
                 "kernel": "k_force_packed<bspline>", "frac": gat_rate / peak,
                 "rel_rms_vs_symmetric": float(torch.sqrt(((acc_g.double() - a32) ** 2).sum() / (a32 ** 2).sum()))}
    del acc_g
    fp64_rate = fp64_pairs / (statistics.mean(fp64_ms) * 1e-3)
    # the paper's tabulated bracket (2^12 NGP bins in r^2) on the same state
    tab_ms = []
    acc_tab = torch.zeros_like(acc)
    for _ in range(3):
        flush.zero_()
        sr.forces_tabulated(pos, 12, acc_tab)
        st = sr.stats()
        tab_ms.append(st.force_kernel_ms)
    tab_err = float(torch.sqrt(((acc_tab.double() - acc64) ** 2).sum() / (acc64 ** 2).sum()))
    tabulated = {"value": st.pairs_last / (statistics.mean(tab_ms) * 1e-3), "unit": UNIT,
                 "kernel_ms": statistics.mean(tab_ms), "rel_rms_vs_fp64": tab_err, "table_entries": 4096}
    # long-range half of the P3M force on the mesh of Eq. phi_gridsize_preference (n_phi = 2 cbrt N)
    from paper_2112_01508_gb300 import LongRange
    long_range = {}
    for prec in (32, 64):
        with LongRange.from_workload(w, precision=prec, device=dev) as lr:
            out = torch.empty((3, n), dtype=torch.float32 if prec == 32 else torch.float64, device=dev)
            for _ in range(2):
                lr.accel(pos, out)
            ts, phases = [], []
            for _ in range(5):
                flush.zero_()
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                lr.accel(pos, out)
                e1.record(stream)
                st_pm = lr.stats()
                ts.append(e0.elapsed_time(e1))
                phases.append(st_pm)
            if prec == 64:
                lr64 = out.clone()
            else:
                lr32 = out.clone()
            long_range[f"fp{prec}"] = {
                "ms": statistics.mean(ts), "n_phi": st_pm.n_phi, "p_i": 2, "p_d": 4,
                "assign_ms": statistics.mean(x.assign_ms for x in phases),
                "fft_ms": statistics.mean(x.fft_ms for x in phases),
                "green_ms": statistics.mean(x.kernel_ms for x in phases),
                "ifft_ms": statistics.mean(x.ifft_ms for x in phases),
                "interp_ms": statistics.mean(x.interp_ms for x in phases),
                "mesh_bytes": st_pm.mesh_bytes, "fft_work_bytes": st_pm.fft_work_bytes}
    long_range["fp32_vs_fp64_rel_rms"] = float(torch.sqrt(((lr32.double() - lr64) ** 2).sum() / (lr64 ** 2).sum()))
    del lr32, lr64
    # the differentiable path: 16 KDK steps with checkpoints every 4 (FP32 forces), then
    # the backward pass (recomputed segments + the adjoint kernel); rung-0 step of Eq. rung
    from paper_2112_01508_gb300.autograd import leapfrog
    dt_lf = (2.0 * eta * w.eps / max(q99, 1e-30)) ** 0.5
    x0 = pos0.clone().requires_grad_(True)
    wts = torch.randn((3, n), dtype=torch.float64, device=dev)
    lf = []
    for _ in range(2):
        x0.grad = None
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e2 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        x16, _ = leapfrog(x0, torch.zeros_like(pos0), sr, dt_lf, 16, 4, precision=32)
        e1.record(stream)
        (x16 * wts).sum().backward()
        e2.record(stream)
        torch.cuda.synchronize()
        lf.append((e0.elapsed_time(e1), e1.elapsed_time(e2)))
    differentiable = {"steps": 16, "checkpoint_every": 4, "precision": "fp32 forces and adjoint",
                      "forward_ms": lf[-1][0], "backward_ms": lf[-1][1],
                      "backward_over_forward": lf[-1][1] / lf[-1][0]}
    del x0, x16, wts
    # substeps of the rung cycle on this state's rungs: receivers l >= l_cur (Section 2.2.2)
    rung_substeps = {}
    for lc in range(n_rung):
        ts, tk = [], []
        for _ in range(3):
            flush.zero_()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            sr.sort(pos, carry=[mom, rung], scratch=scratch)
            sr.build_pairs(None if lc == 0 else rung, lc)
            sr.forces(pos, 32, acc)
            sr.kick(mom, acc, [0.0] * n_rung, rung, lc)  # zero kick: timed, state unchanged
            e1.record(stream)
            st = sr.stats()
            ts.append(e0.elapsed_time(e1))
            tk.append(st.force_kernel_ms)
        rung_substeps[str(lc)] = {"receivers": st.n_active, "pairs": st.pairs_last,
                                  "substep_ms": statistics.mean(ts), "force_kernel_ms": statistics.mean(tk),
                                  "kernel_frac": st.pairs_last / (statistics.mean(tk) * 1e-3) / peak}
    # one global step of the full rung cycle (2^(n_rung-1) substeps, synchronised at its end)
    from paper_2112_01508_gb300.integrate import rung_leapfrog

    def one_cycle(resort_every):
        cyc = {}
        for run in ("timed", "counted"):
            pc, qc = pos0.clone(), torch.zeros_like(mom)
            cyc_pairs = [0]

            def count(k, lmin):
                cyc_pairs[0] += sr.stats().pairs_last
            flush.zero_()
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            rung_leapfrog(sr, pc, qc, dt, eta, w.eps, 1, precision=32, resort_every=resort_every,
                          on_substep=count if run == "counted" else None)
            e1.record(stream)
            torch.cuda.synchronize()
            cyc[run] = (e0.elapsed_time(e1), cyc_pairs[0])
        return {"value": cyc["counted"][1] / (cyc["timed"][0] * 1e-3), "unit": UNIT,
                "ms_per_global_step": cyc["timed"][0], "substeps": 2 ** (n_rung - 1),
                "pairs_per_global_step": cyc["counted"][1], "resort_every": resort_every}

    rung_cycle = one_cycle(4)
    rung_cycle["note"] = ("fake kick + 128 substeps (drift, sort every 4th substep, work list, FP32 forces of due "
                          "rungs, rung kick fused with the next drift)")
    rung_cycle["periodic_resort"] = [one_cycle(k) for k in (1, 16)]
    # subtiles per tile (Section 2.1.3 "Subtiles"; the paper compares fixed 1^3 ... 9^3)
    sweep = {}
    pos_s = pos.clone()
    for ns in (1, 2, 3, 4):
        with ShortRange.from_workload(w, device=dev, n_sub=ns) as s2:
            s2.sort(pos_s)
            s2.build_pairs()
            ts = []
            for _ in range(3):
                flush.zero_()
                s2.forces(pos_s, 32, acc_tab)
                ts.append(s2.stats().force_kernel_ms)
            sweep[str(ns)] = statistics.mean(ts)
    # temporal subtile refinement (trial of one more subdivision every 16 force calls)
    from paper_2112_01508_gb300.refine import SubtileRefiner
    with ShortRange.from_workload(w, device=dev, n_sub=1) as s2:
        ref = SubtileRefiner(s2, interval=16, max_sub=4)
        for _ in range(64):
            ref.before_sort()
            s2.sort(pos_s)
            s2.build_pairs()
            s2.forces(pos_s, 32, acc_tab)
            ref.after_forces()
        refinement = {"start_n_sub": 1, "final_n_sub": ref.current[0], "force_calls": 64, "interval": 16,
                      "trials": [{"n_sub": e[1][0], "record_ps_per_pair": e[2] * 1e9,
                                  "trial_ps_per_pair": e[3] * 1e9, "kept": e[4]} for e in ref.log.events]}
    # per-region refinement: 4 slab regions of the box, each with its own subtiles per
    # tile chosen by the same timed trial rule (Section 2.1.3, "Subtiles": per domain),
    # against every region at a uniform n_sub = 1 ... 4 in the same pipeline
    from paper_2112_01508_gb300.refine import RegionRefiner
    from paper_2112_01508_gb300.slabs import EmulatedSlabs

    def make_region(m):
        return ShortRange(max(m, 1), w.x_s, w.x_r, w.G_m, softening="bspline", eps=w.eps, n_sub=1, device=dev)

    def region_kernel_ms(em, calls=5):
        em.forces(32)  # the first call after a change of decomposition sorts into it
        ts = []
        for _ in range(calls):
            em.forces(32)
            ts.append(sum(rk.stats().force_kernel_ms for rk in em.ranks))
        return statistics.mean(ts)
    regions = {"regions": 4, "force_calls": 64, "interval": 16, "kernel": "k_force_packed<bspline> per region "
               "(receivers: the region's particles; suppliers: region + one-column halo)"}
    em = EmulatedSlabs(pos_s, make_region, 4, n_subs=[1, 1, 1, 1])
    regions["bounds"] = em.bounds
    rr = RegionRefiner(em.ranks, interval=16, max_sub=4)
    for _ in range(64):
        rr.before_sort()
        em.forces(32)
        rr.after_forces()
    rr.before_sort()
    regions["chosen_n_sub"] = [c[0] for c in rr.current]
    regions["chosen_ms"] = region_kernel_ms(em)
    regions["trials"] = [[{"n_sub": e[1][0], "kept": e[4]} for e in log.events] for log in rr.logs]
    uni = {}
    for ns in (1, 2, 3, 4):
        for rk in em.ranks:
            rk.set_subtiles(ns)
        uni[str(ns)] = region_kernel_ms(em)
    regions["uniform_ms"] = uni
    em.close()
    del pos_s

    # end to end through the public API with host buffers: every step's positions and
    # momenta come from pinned host memory and its accelerations go back to it.  The
    # copies run on a second stream, double-buffered, so that the inputs of step k+1
    # and the outputs of step k-1 move while step k computes (each upload is preceded
    # by the 256 MB L2 flush, on the copy stream).
    copy_stream = torch.cuda.Stream(dev)
    P = [pos, torch.empty_like(pos)]
    Q = [mom, torch.empty_like(mom)]
    R = [rung, torch.empty_like(rung)]
    A = [acc, torch.empty_like(acc)]
    copied = [torch.cuda.Event() for _ in range(2)]
    done = [torch.cuda.Event() for _ in range(2)]
    read = [torch.cuda.Event() for _ in range(2)]
    pos_host.copy_(pos0.cpu())
    mom_host.zero_()

    def upload(i):
        with torch.cuda.stream(copy_stream):
            flush.zero_()
            P[i].copy_(pos_host, non_blocking=True)
            Q[i].copy_(mom_host, non_blocking=True)
            copied[i].record(copy_stream)

    S = [[torch.empty_like(pos), torch.empty_like(mom), torch.empty_like(rung)] for _ in range(2)]

    def step_on(i):
        sr.sort(P[i], carry=[Q[i], R[i]], scratch=S[i])
        sr.build_pairs()
        sr.forces(P[i], 32, A[i])
        sr.kick_drift(P[i], Q[i], A[i], R[i], dt, eta, w.eps, kick_factor, drift_factor)

    e_start = torch.cuda.Event(enable_timing=True)
    e_end = torch.cuda.Event(enable_timing=True)
    total_steps = args.warmup + args.steps
    torch.cuda.synchronize()
    for i in range(2):
        read[i].record(copy_stream)
        done[i].record(stream)
    if args.warmup == 0:
        e_start.record(copy_stream)
    upload(0)
    for k in range(total_steps):
        i = k % 2
        stream.wait_event(copied[i])
        stream.wait_event(read[i])          # A[i] of step k-2 has been read back
        step_on(i)
        done[i].record(stream)
        if k + 1 < total_steps:             # inputs of step k+1, once step k-1 released them
            copy_stream.wait_event(done[1 - i])
            if k + 1 == args.warmup:
                e_start.record(copy_stream)
            upload(1 - i)
        copy_stream.wait_event(done[i])     # outputs of step k
        with torch.cuda.stream(copy_stream):
            acc_host.copy_(A[i], non_blocking=True)
            read[i].record(copy_stream)
    e_end.record(copy_stream)
    torch.cuda.synchronize()
    e2e_pairs_step = sr.stats().pairs_last  # every step starts from the same host state
    e2e_total = max_over_ranks(e_start.elapsed_time(e_end), world)
    e2e_value = sum_over_ranks(float(e2e_pairs_step * args.steps), world) / (e2e_total * 1e-3)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        rate, secs, cp, nrecv, cores = cpu_oracle_rate(w, pos_np, args.cpu_sample)
        import oracle
        oracle.set_num_threads(1)
        rate1, secs1, cp1, nrecv1, _ = cpu_oracle_rate(w, pos_np, max(args.cpu_sample // 16, 1))
        oracle.set_num_threads(cores)
        cpu = {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"{nrecv} seeded receivers of the {w.n}-particle set (all suppliers), {cp} pairs, "
                         f"{secs:.1f} s wall",
               "single_core": {"value": rate1, "unit": UNIT, "cores": 1,
                               "sample": f"{nrecv1} seeded receivers, {cp1} pairs, {secs1:.1f} s"}}

    sr.close()
    del flush, P, Q, R, A, S, scratch, pos0, acc64
    torch.cuda.empty_cache()
    large = {}
    if world == 1 and not args.no_large:
        for name in ("n134m", "n1g"):
            large[name] = large_record(name, dev, rank == 0 and not args.no_cpu_baseline)
            torch.cuda.empty_cache()
    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": f"{w.name}: {w.description}", "n": n, "n_sub": w.n_sub,
                       "softening": "bspline", "precision": "fp32 forces, fp64 positions/kicks",
                       "step": "sort+carry, work list, FP32 forces, rungs+kick+drift (one pass; all active)",
                       "l2": "flushed between timed steps (256 MB write)",
                       "parallelism": f"replicas x{world}" if world > 1 else "single GPU"},
            "pairs_per_step": pairs_avg,
            "fp64": {"value": fp64_rate, "unit": UNIT, "kernel_ms": statistics.mean(fp64_ms)},
            "fp32_over_fp64": achieved / fp64_rate,
            "fp32_vs_fp64_rel_rms": parity_32_64,
            "adjoint_over_forward": statistics.mean(vjp_ms) / statistics.mean(fwd_ms),
            "adjoint_over_one_sided_forward": statistics.mean(vjp_ms) / statistics.mean(gat_ms),
            "one_sided_fp32": one_sided,
            "tabulated_2p12": tabulated,
            "n_sub_sweep_force_ms": sweep,
            "long_range_pm": long_range,
            "differentiable_leapfrog": differentiable,
            "subtile_refinement": refinement,
            "subtile_refinement_per_region": regions,
            "rung_substeps": rung_substeps,
            "rung_cycle": rung_cycle,
            "large_workloads": large,
            "roofline": roofline,
            "hbm": hbm,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": 2 * 3 * 8 * n,
                    "d2h_bytes_per_step": 3 * 4 * n, "ms_per_step": e2e_total / args.steps,
                    "copies": "pinned host buffers, double-buffered on a second stream, overlapped with compute"},
            "gpu_launches": launches,
            "clocks": clocks,
            "wall_s_timed": t_wall,
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def run_slabs(args):
    """The sharded path: each rank owns a work-balanced slab of tile columns of the 128^3
    set; per step it sorts its particles, exchanges emigrants and the one-column halo with
    its two neighbours (NCCL send/recv into its own memory), sorts particles plus halo,
    computes the FP32 forces of its own particles and applies rungs, kick and drift.
    Strong scaling: the whole set is fixed, value = pairs over all ranks / slowest rank."""
    import torch

    import synth
    from paper_2112_01508_gb300 import ShortRange
    from paper_2112_01508_gb300.slabs import DistTransport, SlabExchange, SlabRank, initial_split

    world, rank, local = dist_setup()
    dev = torch.device("cuda", local)
    w = synth.workload(args.workload)
    n = w.n
    eta, n_rung = 0.025, 8
    pos = torch.from_numpy(synth.workload_positions(w)).to(dev)  # every rank draws the same set
    mom = torch.zeros((3, n), dtype=torch.float64, device=dev)
    rung = torch.zeros(n, dtype=torch.int8, device=dev)

    def make(m):
        return ShortRange(max(m, 1), w.x_s, w.x_r, w.G_m, softening="bspline", eps=w.eps, n_sub=w.n_sub,
                          device=dev)
    with make(n) as full:
        # time step from the fake kick on the whole set, as in the single-GPU benchmark
        full.sort(pos)
        full.build_pairs()
        a64 = full.forces(pos, 64)
        amag = torch.linalg.vector_norm(a64, dim=0)
        q99 = float(torch.quantile(amag[torch.randperm(n, device=dev, generator=torch.Generator(device=dev).manual_seed(0))[:1 << 20]].float(), 0.99))
        del a64, amag
        bounds, parts = initial_split(full, pos, [mom, rung], world)
        n_t = full.stats_geometry()[0]
    del pos, mom, rung
    dt = 64.0 * (2.0 * eta * w.eps / max(q99, 1e-30)) ** 0.5
    kick_factor = [dt / 2 ** l for l in range(n_rung)]
    ex = SlabExchange(n_t, bounds, rank, world)
    rk = SlabRank(make, ex)
    tr = DistTransport()
    own = parts[rank]
    stream = torch.cuda.current_stream(dev)

    def step(own):
        col = rk.sort_own(own)
        out = ex.prepare(own, col)
        fl, fr = tr.swap(ex, out)
        own, halo = ex.finish(out, fl, fr)
        acc, pairs = rk.forces(own[0], halo, 32)
        rk.kick_drift(own, acc, dt, eta, w.eps, kick_factor, dt / 2 ** (n_rung - 1))
        return own, pairs, halo.shape[1]

    for _ in range(args.warmup):
        own, _, _ = step(own)
    torch.cuda.synchronize()
    barrier(world)
    ms, prs, halos, owns = [], [], [], []
    for _ in range(args.steps):
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        own, pairs, nh = step(own)
        e1.record(stream)
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
        prs.append(pairs)
        halos.append(nh)
        owns.append(own[0].shape[1])
    barrier(world)
    total_ms = max_over_ranks(sum(ms), world)
    total_pairs = sum_over_ranks(float(sum(prs)), world)
    rk.close()
    if rank == 0:
        line = {"metric": METRIC, "value": total_pairs / (total_ms * 1e-3), "unit": UNIT, "n_gpus": world,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": total_ms / args.steps,
                "higher_is_better": True, "scaling": "strong", "vs_baseline": None, "dtype": "f32",
                "data": "synthetic",
                "config": {"workload": f"{w.name}: {w.description}", "n": n, "n_sub": w.n_sub,
                           "softening": "bspline", "parallelism": f"slabs x{world} (tile columns along x, "
                                                                  "one-column halo by NCCL send/recv)",
                           "slab_bounds": bounds,
                           "step": "sort own, exchange emigrants + halo, sort own + halo, FP32 forces of own "
                                   "particles (one-sided), rungs+kick+drift"},
                "rank0": {"own_particles": statistics.mean(owns), "halo_particles": statistics.mean(halos),
                          "ms_per_step": statistics.mean(ms)}}
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def run_only(args):
    """Profiling mode: sort once, then repeat one entry point (for ncu captures)."""
    import torch

    import synth
    from paper_2112_01508_gb300 import ShortRange

    dev = torch.device("cuda", 0)
    w = synth.workload(args.workload)
    pos = torch.from_numpy(synth.workload_positions(w)).to(dev)
    sr = ShortRange.from_workload(w, device=dev)
    sr.sort(pos)
    sr.build_pairs()
    acc32 = torch.zeros((3, w.n), dtype=torch.float32, device=dev)
    acc64 = torch.zeros((3, w.n), dtype=torch.float64, device=dev)
    abar = torch.randn((3, w.n), dtype=torch.float32, device=dev) if args.only == "vjp32" else None
    times = []
    if args.only == "pm32":
        from paper_2112_01508_gb300 import LongRange
        with LongRange.from_workload(w, precision=32, device=dev) as lr:
            for k in range(args.warmup + args.steps):
                lr.accel(pos, acc32)
                st = lr.stats()
                if k >= args.warmup:
                    times.append({"total": st.total_ms, "assign": st.assign_ms, "fft": st.fft_ms,
                                  "green": st.kernel_ms, "ifft": st.ifft_ms, "interp": st.interp_ms})
        print(json.dumps({"only": args.only, "workload": w.name, "mesh_ms": times, "n_phi": w.n_phi}))
        sr.close()
        return
    if args.only == "rung_steps":
        # the full step (all particles receivers) and the deepest-rung substep (~1% of the
        # particles on rung 7 by the fake kick's |a|, Eq. rung), FP32 and FP64 paths
        eta, n_rung = 0.025, 8
        res = {"only": args.only, "workload": w.name, "n": w.n}
        ts = []
        for k in range(args.warmup + args.steps):
            sr.forces(pos, 32, acc32)
            if k >= args.warmup:
                ts.append(sr.stats().force_kernel_ms)
        st = sr.stats()
        res["full_fp32"] = {"kernel_ms": ts, "pairs": st.pairs_last}
        amag = torch.linalg.vector_norm(acc32, dim=0)
        pick = torch.randperm(w.n, device=dev, generator=torch.Generator(device=dev).manual_seed(0))[:1 << 20]
        q99 = float(torch.quantile(amag[pick], 0.99))
        del amag, pick
        dt = 64.0 * (2.0 * eta * w.eps / q99) ** 0.5
        rung = sr.assign_rungs(acc32, dt, eta, w.eps)
        sr.build_pairs(rung, n_rung - 1)
        for prec, out in ((32, acc32), (64, acc64)):
            ts = []
            for k in range(args.warmup + args.steps if prec == 32 else 1):
                sr.forces(pos, prec, out)
                if prec == 64 or k >= args.warmup:
                    ts.append(sr.stats().force_kernel_ms)
            st = sr.stats()
            res[f"deepest_rung_fp{prec}"] = {"kernel_ms": ts, "pairs": st.pairs_last, "receivers": st.n_active}
        print(json.dumps(res))
        sr.close()
        return
    if args.evolve:
        # the state after some benchmark steps (fake-kick step, then sort, forces, rungs+kick+drift)
        mom = torch.zeros((3, w.n), dtype=torch.float64, device=dev)
        rung0 = torch.zeros(w.n, dtype=torch.int8, device=dev)
        sr.forces(pos, 64, acc64)
        amag = torch.linalg.vector_norm(acc64, dim=0)
        gen = torch.Generator(device=dev).manual_seed(0)
        q99 = float(torch.quantile(amag[torch.randperm(w.n, device=dev, generator=gen)[:1 << 20]].float(), 0.99))
        dt = 64.0 * (2.0 * 0.025 * w.eps / q99) ** 0.5
        for _ in range(args.evolve):
            sr.sort(pos, carry=[mom, rung0])
            sr.build_pairs()
            sr.forces(pos, 32, acc32)
            sr.kick_drift(pos, mom, acc32, rung0, dt, 0.025, w.eps, [dt / 2 ** l for l in range(8)], dt / 128)
        sr.sort(pos)
        sr.build_pairs()
        del mom, rung0
    if args.only == "substep":
        # a deep-rung substep: receivers on rung 7 of a fake kick whose step puts ~12% of
        # the particles there (Eq. rung); all particles supply
        sr.forces(pos, 32, acc32)
        amag = torch.linalg.vector_norm(acc32, dim=0)
        gen = torch.Generator(device=dev).manual_seed(0)
        q = float(torch.quantile(amag[torch.randperm(w.n, device=dev, generator=gen)[:1 << 20]], 0.88))
        rung = sr.assign_rungs(acc32, 64.0 * (2.0 * 0.025 * w.eps / q) ** 0.5, 0.025, w.eps)
        sr.build_pairs(rung, 7)
        for k in range(args.warmup + args.steps):
            sr.forces(pos, 32, acc32)
            st = sr.stats()
            if k >= args.warmup:
                times.append(st.force_kernel_ms)
        print(json.dumps({"only": args.only, "workload": w.name, "kernel_ms": times, "pairs": st.pairs_last,
                          "receivers": st.n_active, "chunks": st.n_chunks}))
        sr.close()
        return
    if args.only == "kick":
        # Eq. rung + kick + drift in one pass (p3m_sr_kick_drift) on the 128^3 state
        mom = torch.zeros((3, w.n), dtype=torch.float64, device=dev)
        rung = torch.zeros(w.n, dtype=torch.int8, device=dev)
        sr.forces(pos, 32, acc32)
        stream = torch.cuda.current_stream(dev)
        dt = 1e-4
        kf = [dt / 2 ** l for l in range(8)]
        for k in range(args.warmup + args.steps):
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            sr.kick_drift(pos, mom, acc32, rung, dt, 0.025, w.eps, kf, dt / 128)
            e1.record(stream)
            torch.cuda.synchronize()
            if k >= args.warmup:
                times.append(e0.elapsed_time(e1))
        print(json.dumps({"only": args.only, "workload": w.name, "kernel_ms": times}))
        sr.close()
        return
    if args.only == "forces32_gather":
        sr.set_symmetric(False)
    for k in range(args.warmup + args.steps):
        if args.only in ("forces32", "forces32_gather"):
            sr.forces(pos, 32, acc32)
        elif args.only == "forces64":
            sr.forces(pos, 64, acc64)
        elif args.only == "vjp32":
            sr.vjp(pos, abar, 32)
        else:
            sr.sort(pos)
        st = sr.stats()
        if k >= args.warmup:
            times.append(st.vjp_kernel_ms if args.only == "vjp32" else st.force_kernel_ms)
    print(json.dumps({"only": args.only, "workload": w.name, "kernel_ms": times, "pairs": st.pairs_last}))
    sr.close()


def run_reference(args):
    """The reference arm: the CPU oracle as it stands on the host cores."""
    import synth

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    w = synth.workload(args.workload)
    pos = synth.workload_positions(w)
    ts, ps = [], []
    cores = 1
    for k in range(args.warmup + args.steps):
        rate, secs, pairs, nrecv, cores = cpu_oracle_rate(w, pos, args.ref_sample, seed=100 + k)
        if k >= args.warmup:
            ts.append(secs)
            ps.append(pairs)
    value = sum(ps) / sum(ts)
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * sum(ts) / len(ts), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": f"{w.name}: {w.description}", "n": w.n, "softening": "bspline"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": f"{args.ref_sample} seeded receivers per step, all {w.n} suppliers"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def main():
    args = parse_args()
    if args.impl == "reference":
        run_reference(args)
    elif args.only:
        run_only(args)
    elif args.mode == "slabs":
        run_slabs(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
