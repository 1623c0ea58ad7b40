#!/usr/bin/env python
"""Throughput benchmark of the GB300 PIMD path (bead-atom-steps/s).

Workload (the plain FP64 configuration): a flexible water-like box of 64
molecules (192 atoms) in a 12.42 A periodic box, P = 32 beads, T = 300 K,
dt = 0.5 fs, BAOAB with PILE_L, FP64.  One benchmark step is 1000 MD steps
with the App. A estimators reduced and copied to the host every 100 steps.
Inputs are synthetic (seeded placement, see paper_2602_13553_gb300.inputs).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Prints one JSON line on rank 0.  Under torchrun (N > 1) every rank advances
its own independent replica (different seed) with no data-path collective:
weak scaling, replicas only.  ``--impl reference`` times the CPU oracle on the
host cores instead (rank 0 only).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

WORKLOAD = dict(nmol=64, L=12.42, P=32, T=300.0, dt=5e-4, md_per_step=1000, est_every=100,
                tau=1.0)
WORKLOAD_NAME = ("water-like box, 64 molecules (192 atoms), 12.42 A periodic, P=32 beads, "
                 "T=300 K, dt=0.5 fs, BAOAB+PILE_L, FP64")
METRIC = "bead-atom-steps/s"
FP64_NOMINAL = 152 * 4 * 2.07e9  # 152 SMs x 2 FP64 FMA/clk x 2 flop x 2.07 GHz (context only)
L2_FLUSH_BYTES = 512 << 20


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=60)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--fp64-steps", type=int, default=None,
                    help="timed steps of the plain FP64 workload (default: --steps)")
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--no-sweep", action="store_true")
    ap.add_argument("--no-serve", action="store_true")
    ap.add_argument("--batched-steps", type=int, default=20)
    ap.add_argument("--serve-jobs", type=int, default=2000)
    ap.add_argument("--serve-step-scale", type=float, default=1.0)
    return ap.parse_args()


def dist_env():
    return (int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")),
            int(os.environ.get("LOCAL_RANK", "0")))


def barrier(world):
    """Host barrier across the replica ranks (gloo; no data-path collective)."""
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x, world):
    """The slowest rank's elapsed time: every rank's value, maximum taken."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(world, units_per_rank, seconds):
    """Whole-job throughput: the units all ranks processed over the slowest
    rank's time (weak scaling: every rank holds its own replica)."""
    return world * units_per_rank / seconds


def system(seed):
    from paper_2602_13553_gb300 import inputs
    w = WORKLOAD
    x0, mass = inputs.water_box(w["nmol"], w["L"], w["P"], seed, jitter=0.02)
    return x0, mass, dict(T=w["T"], dt=w["dt"], potential=1, ff=inputs.WATER_FF,
                          box=(w["L"],) * 3, seed=seed, tau=w["tau"])


def config(extra=None):
    w = WORKLOAD
    c = {"workload": WORKLOAD_NAME, "atoms": 3 * w["nmol"], "beads": w["P"],
         "md_steps_per_bench_step": w["md_per_step"], "estimators_every": w["est_every"],
         "l2": "flushed (512 MiB write) between timed steps; state 0.44 MB < L2",
         "data": "synthetic"}
    if extra:
        c.update(extra)
    return c


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.proc = None
        self.gpu = gpu_index
        self.path = os.path.join(tempfile.gettempdir(), "pimd_bench_clocks_%d.csv" % os.getpid())

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                 "-lms", "100", "-i", str(self.gpu)], stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.f.close()
        sm, mx, reasons = [], [], set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "samples": len(sm),
                "reasons": sorted(reasons)}


def step_flops_per_bead_atom(P):
    """Algorithmic FP64 flops of the fused step kernel per bead-atom: three
    folded normal-mode transforms of 3 components, each output a sum over one
    half of its folded row (P/2 + 1 FMAs: 9 P + 18), the folding and
    recombination adds (9), the merged kick (6), two exact rotations (36) and
    the O update (9); the Box-Muller noise is not counted.  The kernel takes
    the sums in fixed point on the integer pipe, so this rate can exceed the
    FP64 pipe's."""
    return 9 * P + 78


# 32 x 32 -> 64-bit integer multiply-adds of a GB300 a second (eight independent
# chains a thread, four blocks of 256 threads an SM, measured): the rate that
# the fixed-point transforms of the FP64 step are held against
INT_MAD_RATE = 18.1e12


def well_step_mads_per_bead_atom(P):
    """Integer multiply-adds of the FP64 step kernel per bead-atom in a harmonic
    well, where F~ = -k q~ leaves two transforms of 3 components: an output is a
    sum over one half of its folded row in pairs of terms, three multiply-adds a
    product (28-bit limbs).  Noise and scalings are not counted."""
    return 2 * 3 * 3 * 2 * ((P // 2 + 2) // 2)


def force_flops(x, L, rc, rlist):
    """Algorithmic FP64 flops of one water force launch (all beads) for the
    positions x [P][N][3]: 30 per O-O pair inside rc, each unordered pair
    counted once (minimum-image distance, Lennard-Jones force, energy and
    virial), and 120 per molecule and bead for the two bonds and the angle --
    about 200 per bead-atom at 1 g/cm^3 and rc = 6 A.  Returned with the
    overhead that is not the method's work: 17 flops per neighbour-list
    candidate (centroid pair within rc + skin) and bead, the distance tests
    of pairs that turn out to lie beyond rc."""
    P = x.shape[0]
    O = x[:, 0::3, :]
    nmol = O.shape[1]
    cen = O.mean(axis=0)
    d = cen[None, :, :] - cen[:, None, :]
    d -= L * np.rint(d / L)
    cand = ((np.einsum("ijk,ijk->ij", d, d) < rlist * rlist).sum() - nmol) // 2
    inside = 0
    for k in range(P):
        e = O[k][None, :, :] - O[k][:, None, :]
        e -= L * np.rint(e / L)
        inside += ((np.einsum("ijk,ijk->ij", e, e) < rc * rc).sum() - nmol) // 2
    return 30.0 * inside + 120.0 * nmol * P, 17.0 * cand * P


def hbm_peak():
    """Measured copy bandwidth of this GPU pool (GB/s), else the fallback."""
    try:
        return float(json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


SWEEP = ((1 << 20, 8), (1 << 18, 32), (1 << 17, 64), (1 << 16, 128))


def sweep_bench(stream, steps=4, warmup=2):
    """The oscillator throughput sweep: N independent 3D oscillators (m = 1.008
    amu, hbar omega = 0.1 eV, 300 K, dt = 0.25 fs, PILE_L) with N P = 2^23
    bead-atoms (201 MB of FP64 state, beyond the 129 MB L2) for P = 8, 32,
    64, 128, in FP64 and in split precision.  Per point: bead-atom-steps/s
    over `steps` calls of 10 MD steps (CUDA events on the library's stream)
    and the roofline of the step kernel, from its own CUDA-event time per
    launch: FP64 against the integer pipe, which holds its transforms
    (well_step_mads_per_bead_atom), split against HBM (48 B + 96 B / P per
    bead-atom: deviations and velocities read and written, no forces; the
    centroids)."""
    import torch
    from paper_2602_13553_gb300 import binding, inputs
    hbar = 4.135667403e-3 / (2 * math.pi)
    omega = 0.1 / hbar
    hbm, hsrc = hbm_peak()
    out = []
    for N, P in SWEEP:
        x0, mass = inputs.harmonic(N, P, seed=1, std=0.1)
        for prec, name in ((0, "fp64"), (1, "split")):
            sim = binding.Simulation(x0, mass, T=300.0, dt=2.5e-4, potential=0, ff=(omega,),
                                     precision=prec, stream=stream.cuda_stream)
            for _ in range(warmup):
                sim.step(10)
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            for _ in range(steps):
                sim.step(10)
            e1.record(stream)
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1)
            sim.set_kernel_timing(True)
            sim.step(10)
            kt = sim.kernel_times()
            sim.set_kernel_timing(False)
            step_ms = kt["step"][0] / max(1, kt["step"][1])
            units = N * P
            pt = {"N": N, "P": P, "precision": name, "value": units * 10 * steps / (ms / 1e3),
                  "step_kernel_ms": step_ms}
            if prec == 0:
                ach = well_step_mads_per_bead_atom(P) * units / (step_ms / 1e3) / 1e12
                pt["roofline"] = {"bound": "alu", "achieved": ach, "peak": INT_MAD_RATE / 1e12,
                                  "unit": "T 32-bit multiply-adds/s", "frac": ach / (INT_MAD_RATE / 1e12),
                                  "peak_source": "measured 32 x 32 -> 64-bit multiply-add throughput"}
            else:
                ach = (48.0 + 96.0 / P) * units / (step_ms / 1e3) / 1e9
                pt["roofline"] = {"bound": "hbm", "achieved": ach, "peak": hbm, "unit": "GB/s",
                                  "frac": ach / hbm, "peak_source": hsrc}
            out.append(pt)
            sim.close()
            del sim
    return {"workload": "N 3D oscillators, N P = 2^23 bead-atoms, 300 K, dt 0.25 fs, PILE_L",
            "unit": METRIC, "points": out}


def same_mix_handles(reps, precision, md_steps=100, warm=10):
    """The replicas of the batched mix as independent single-system handles
    (plain FP64 or split precision), each on its own CUDA stream, all
    stepped together: bead-atom-steps/s of md_steps steps (host clock around
    the launches and a device synchronise)."""
    import torch
    from paper_2602_13553_gb300 import binding, inputs
    sims, streams = [], []
    units = 0
    for r in reps:
        x0, mass = inputs.water_box(r.nmol, r.L, r.P, r.seed, jitter=0.02, deuterium=r.deuterium)
        st = torch.cuda.Stream()
        sims.append(binding.Simulation(x0, mass, T=r.T, dt=5e-4, potential=binding.POT_WATERLIKE,
                                       ff=inputs.water_ff_for_box(r.L), box=(r.L,) * 3, seed=r.seed,
                                       precision=precision, stream=st.cuda_stream))
        streams.append(st)
        units += 3 * r.nmol * r.P
    for sim in sims:
        sim.step(warm)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for sim in sims:
        sim.step(md_steps)
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    for sim in sims:
        sim.close()
    return units * md_steps / dt


def batched_bench(stream, steps, warmup):
    """The batched workload: 256 independent water-like replicas (32-512
    molecules log-uniform at 1 g/cm^3, P in {8,16,32,64}, T in [100,400] K,
    H or D), split precision, one batch; each timed step is 100 MD steps of
    every replica plus the estimators of all of them."""
    import torch
    from paper_2602_13553_gb300 import binding, inputs
    reps = inputs.replica_mix(256, seed=1)
    b = binding.Batch(256, stream=stream.cuda_stream)
    units = 0
    step_bytes = 0.0
    force_bytes = 0.0
    md_bytes = 0.0
    for r in reps:
        x0, mass = inputs.water_box(r.nmol, r.L, r.P, r.seed, jitter=0.02, deuterium=r.deuterium)
        b.add(x0, mass, T=r.T, dt=5e-4, nsteps=10 ** 12, ff=inputs.water_ff_for_box(r.L),
              box=(r.L,) * 3, seed=r.seed)
        N = 3 * r.nmol
        units += N * r.P
        # compulsory HBM bytes per launch: step reads d, v~, F and writes d, v~
        # (FP32, 60 B per bead-atom) plus 124 B per atom (FP64 centroid position
        # and velocity read+write, wrapped FP32 centroid, two FP64 constants);
        # force reads d and writes F (24 B per bead-atom), 12 B per atom of
        # centroids, 16 B per molecule-bead of energy/virial rows
        step_bytes += 60.0 * N * r.P + 124.0 * N
        force_bytes += 24.0 * N * r.P + 12.0 * N + 16.0 * r.nmol * r.P
        # the whole split-precision MD step's compulsory bytes: 84 B per
        # bead-atom + 120 B per atom (FP64 centroid x, v~_0 read and written)
        md_bytes += 84.0 * N * r.P + 120.0 * N
    tiles = b.autotune(3)
    for _ in range(warmup):
        b.run(100)
        b.estimators()
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    l0 = b.kernel_launches()
    for i in range(steps):
        ev[i][0].record(stream)
        b.run(100)
        b.estimators()
        ev[i][1].record(stream)
    torch.cuda.synchronize()
    launches = b.kernel_launches() - l0
    ms = sum(a.elapsed_time(c) for a, c in ev)
    value = units * 100.0 * steps / (ms / 1e3)
    stp, _, rb = b.status(rebuilds=True)
    live = stp >= 0
    rebuild_rate = float(rb[live].sum() / max(1, stp[live].sum()))
    kt = b.time_kernels(10)
    # the transform A/B: the same replicas on the block-item kernel with FP32
    # FMA transforms (default tiles), step kernels timed the same way
    b.set_transforms("ffma")
    b.run(20)
    kt_ffma = b.time_kernels(10)
    b.set_transforms("tensor")
    dom = "step" if kt["step"] >= kt["force"] else "force"
    per_ms = kt[dom] / 10.0
    bytes_ = step_bytes if dom == "step" else force_bytes
    peak, src = hbm_peak()
    achieved = bytes_ / (per_ms / 1e3) / 1e9
    md_ms = ms / steps / 100.0          # per MD step, estimators included
    b.close()
    tot = sum(kt.values())
    return {
        "workload": "256 water-like replicas, 32-512 molecules log-uniform, P in {8,16,32,64}, "
                    "T 100-400 K, H/D, split precision",
        "value": value, "unit": METRIC, "ms_per_step": ms / steps, "md_steps_per_step": 100,
        "bead_atoms": units, "steps": steps, "gpu_launches": int(launches), "dtype": "f32+f64 split",
        "autotuned_tiles": {str(k): v for k, v in tiles.items()},
        "nbr_rebuilds_per_replica_step": rebuild_rate,
        "vs_plain_fp64": None,
        "roofline": {"bound": "hbm", "kernel": "k_bstep_w" if dom == "step" else "k_bforce",
                     "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                     "peak_source": src, "algorithmic_bytes_per_launch": bytes_,
                     "avg_launch_ms": per_ms,
                     "kernel_time_share": {k: round(v / tot, 4) for k, v in kt.items()}},
        "same_mix": {"plain_fp64_handles": same_mix_handles(reps, 0), "split_handles": same_mix_handles(reps, 1),
                     "unit": METRIC,
                     "basis": "the same 256 replicas as independent single-system handles, one CUDA stream "
                              "each, 100 MD steps of all of them (host clock around launches and a device "
                              "synchronise): plain FP64, and split precision without the batch engine"},
        "transform_ab": {"tensor_core_step_ms": kt["step"] / 10.0, "ffma_step_ms": kt_ffma["step"] / 10.0,
                         "basis": "per-MD-step device time of the step kernels over the mix: warp items with "
                                  "3xTF32 mma.sync transforms against block items with FP32 FMA transforms"},
        "whole_step": {"bound": "hbm", "achieved": md_bytes / (md_ms / 1e3) / 1e9, "peak": peak,
                       "unit": "GB/s", "frac": md_bytes / (md_ms / 1e3) / 1e9 / peak, "peak_source": src,
                       "algorithmic_bytes_per_md_step": md_bytes, "ms_per_md_step": md_ms,
                       "basis": "84 B per bead-atom + 120 B per atom per MD step over the "
                                "measured time of an MD step (estimators every 100 included)"},
    }


def serve_bench(stream, n_jobs, step_scale):
    """The serving workload: a Poisson stream of water-like jobs at 50 jobs/s
    (96-12288 atoms, P 4-128, 1k-50k steps, all log-uniform) against a 150 GB
    budget; the first n_jobs of the trace (by default all 2000), step counts
    scaled by step_scale (by default 1)."""
    from paper_2602_13553_gb300 import binding, inputs
    trace = inputs.serving_trace(n_jobs, 50.0, seed=1)
    srv = binding.Server(150 * 10 ** 9, max_replicas=512, chunk_steps=100, stream=stream.cuda_stream)
    ids = []
    t0 = time.perf_counter()
    for j in trace:
        # each job's box is drawn just before its arrival time (milliseconds),
        # then submitted at that time
        L = inputs.box_length(j.nmol)
        x0, mass = inputs.water_lattice_box(j.nmol, L, j.P, j.seed % (2 ** 31), jitter=0.02)
        n = max(1, int(round(j.nsteps * step_scale)))
        delay = j.arrival_s - (time.perf_counter() - t0)
        if delay > 0:
            time.sleep(delay)
        ids.append(srv.submit(x0, mass, T=j.T, dt=5e-4, nsteps=n, ff=inputs.water_ff_for_box(L),
                              box=(L,) * 3, seed=j.seed))
    pending = set(ids)
    while pending:
        for jid in list(pending):
            if srv.poll(jid) is not None:
                pending.discard(jid)
        time.sleep(0.01)
    lat, first, last = [], None, None
    for jid in ids:
        sub, start, end = srv.times(jid)
        lat.append(end - sub)
        first = sub if first is None else min(first, sub)
        last = end if last is None else max(last, end)
    st = srv.stats()
    srv.close()
    lat = np.array(lat)
    return {
        "workload": ("Poisson water-like jobs at 50/s, 96-12288 atoms, P 4-128, 1k-50k steps (log-uniform), "
                     "first %d jobs of the trace, steps x %g" % (n_jobs, step_scale)),
        "jobs": n_jobs, "completed": int(st["completed"]), "failed": int(st["failed"]),
        "p50_ms": float(np.percentile(lat, 50) * 1e3), "p99_ms": float(np.percentile(lat, 99) * 1e3),
        "aggregate": st["bead_atom_steps"] / (last - first), "unit": METRIC,
        "makespan_s": last - first, "gpu_busy_s": st["gpu_busy_s"], "chunks": int(st["chunks"]),
        "hbm_budget_gb": 150,
    }


def cpu_baseline(target_s=12.0):
    """The CPU oracle as it stands, on the host cores, on a bounded sample of
    the same workload (MD steps of the same system, estimators every 100)."""
    import oracle
    ncores = os.cpu_count() or 1
    oracle.set_threads(ncores)
    x0, mass, kw = system(1)
    sim = oracle.Sim(x0, mass, **kw)
    w = WORKLOAD
    t0 = time.perf_counter()
    sim.run(20)
    probe = time.perf_counter() - t0
    n = int(max(20, min(5000, target_s / max(probe / 20, 1e-6))))
    n = max(100, (n // 100) * 100)
    t0 = time.perf_counter()
    done = 0
    while done < n:
        sim.run(w["est_every"])
        sim.estimators()
        done += w["est_every"]
    dt = time.perf_counter() - t0
    value = 3 * w["nmol"] * w["P"] * n / dt
    return {"value": value, "unit": METRIC, "cores": oracle.max_threads(), "kind": "oracle",
            "sample": "%d MD steps (estimators every 100) of the same 192-atom x 32-bead system, "
                      "%.1f s wall" % (n, dt)}


def _time_oracle(sim, units_per_step, chunk, budget_s, with_est):
    """Bead-atom-steps/s of the oracle on `sim` over about budget_s seconds
    (whole chunks of `chunk` MD steps, estimators after each if asked)."""
    t0 = time.perf_counter()
    done = 0
    while True:
        sim.run(chunk)
        if with_est:
            sim.estimators()
        done += chunk
        dt = time.perf_counter() - t0
        if dt >= budget_s:
            return units_per_step * done / dt, done, dt


def oracle_configs(budget_s=2.5):
    """The oracle on the other workloads of the study, on all host cores and,
    for the benchmark system, on one core: 64 harmonic oscillators x 8 beads,
    the 192-atom x 32-bead water box, 512 molecules x 64 beads (a few steps
    of it) and one replica of the 256-replica mix (its median size)."""
    import oracle
    from paper_2602_13553_gb300 import inputs
    ncores = os.cpu_count() or 1
    out = []
    hbar = 4.135667403e-3 / (2 * math.pi)

    def rec(name, sim, units, chunk, threads, with_est=True):
        oracle.set_threads(threads)
        v, n, dt = _time_oracle(sim, units, chunk, budget_s, with_est)
        out.append({"config": name, "value": v, "unit": METRIC, "cores": oracle.max_threads(),
                    "sample": "%d MD steps, %.1f s" % (n, dt)})

    x0, mass = inputs.harmonic(64, 8, seed=1, std=0.1)
    rec("64 harmonic oscillators x 8 beads", oracle.Sim(x0, mass, T=300.0, dt=2.5e-4, potential=0,
                                                         ff=(0.1 / hbar,), seed=1), 64 * 8, 100, ncores)
    x0, mass, kw = system(1)
    rec("water-like 192 atoms x 32 beads, one core", oracle.Sim(x0, mass, **kw), 192 * 32, 100, 1)
    rec("water-like 192 atoms x 32 beads", oracle.Sim(x0, mass, **kw), 192 * 32, 100, ncores)
    L2 = inputs.box_length(512)
    x0, mass = inputs.water_box(512, L2, 64, 1, jitter=0.02)
    rec("water-like 1536 atoms x 64 beads", oracle.Sim(x0, mass, T=300.0, dt=5e-4, potential=1,
                                                      ff=inputs.water_ff_for_box(L2), box=(L2,) * 3, seed=1),
        1536 * 64, 2, ncores, with_est=False)
    reps = sorted(inputs.replica_mix(256, 1), key=lambda r: r.nmol * r.P)
    r = reps[len(reps) // 2]
    x0, mass = inputs.water_box(r.nmol, r.L, r.P, r.seed, jitter=0.02, deuterium=r.deuterium)
    rec("median replica of the mix: %d molecules x %d beads" % (r.nmol, r.P),
        oracle.Sim(x0, mass, T=r.T, dt=5e-4, potential=1, ff=inputs.water_ff_for_box(r.L), box=(r.L,) * 3,
                   seed=1), 3 * r.nmol * r.P, 20, ncores)
    oracle.set_threads(ncores)
    return out


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    import oracle
    ncores = os.cpu_count() or 1
    oracle.set_threads(ncores)
    w = WORKLOAD
    x0, mass, kw = system(1)
    sim = oracle.Sim(x0, mass, **kw)
    per = w["est_every"]                 # each reference step: 100 MD steps + estimators
    for _ in range(args.warmup):
        sim.run(per)
        sim.estimators()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        sim.run(per)
        sim.estimators()
    dt = time.perf_counter() - t0
    value = 3 * w["nmol"] * w["P"] * per * args.steps / dt
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": METRIC,
            "n_gpus": 0, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * dt / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": config({"reference_step": "%d MD steps + estimators (bounded sample of the "
                              "1000-step benchmark step)" % per}),
            "cpu_baseline": {"value": value, "unit": METRIC, "cores": oracle.max_threads(),
                             "kind": "oracle",
                             "sample": "%d x %d MD steps of the benchmark system" % (args.steps, per)},
            "e2e": {"value": value, "unit": METRIC, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def run_ours(args):
    import torch
    from paper_2602_13553_gb300 import binding, build
    rank, world, local = dist_env()
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("gloo")
    torch.cuda.set_device(local)
    build.build()
    w = WORKLOAD
    seed = 1 + rank
    x0, mass, kw = system(seed)
    stream = torch.cuda.Stream()
    binding.use_torch_allocator()
    sim = binding.Simulation(x0, mass, stream=stream.cuda_stream, **kw)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device="cuda")
    fp64_peak = binding.fp64_fma_rate()   # TFLOP/s, measured on this GPU before the timed region
    nchunks = w["md_per_step"] // w["est_every"]

    def bench_step():
        for _ in range(nchunks):
            sim.step(w["est_every"])
            sim.estimators()

    def flush_l2():
        with torch.cuda.stream(stream):
            flush.fill_(rank & 0xff)

    for _ in range(max(3, args.warmup)):
        flush_l2()
        bench_step()
    barrier(world)
    torch.cuda.synchronize()
    clocks = Clocks(local)
    clocks.start()
    launches0 = sim.kernel_launches()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    for i in range(args.steps):
        flush_l2()
        ev[i][0].record(stream)
        bench_step()
        ev[i][1].record(stream)
    torch.cuda.synchronize()
    barrier(world)
    launches = sim.kernel_launches() - launches0
    clk = clocks.stop()
    total_ms = max_over_ranks(sum(a.elapsed_time(b) for a, b in ev), world)
    units_per_rank = 3 * w["nmol"] * w["P"] * w["md_per_step"] * args.steps
    value = job_throughput(world, units_per_rank, total_ms / 1e3)

    # --- per-kernel device durations (CUDA events around every launch) -----
    ksteps = min(args.steps, 10)
    sim.set_kernel_timing(True)
    for _ in range(ksteps):
        flush_l2()
        bench_step()
    kt = sim.kernel_times()
    sim.set_kernel_timing(False)
    xs, _, _ = sim.get_state()

    # --- end to end through the C ABI with pinned host buffers -------------
    xh = torch.empty(x0.shape, dtype=torch.float64, pin_memory=True)
    vh = torch.empty(x0.shape, dtype=torch.float64, pin_memory=True)
    xa, va, st0 = sim.get_state()
    xh.numpy()[:] = xa
    vh.numpy()[:] = va
    e2e_steps = max(3, args.steps // 2)
    barrier(world)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        sim.set_state(xh.numpy(), vh.numpy(), st0)
        bench_step()
    torch.cuda.synchronize()
    e2e_s = max_over_ranks(time.perf_counter() - t0, world)
    e2e_value = job_throughput(world, 3 * w["nmol"] * w["P"] * w["md_per_step"] * e2e_steps, e2e_s)
    P, N = w["P"], 3 * w["nmol"]
    h2d = 2 * P * N * 3 * 8
    d2h = nchunks * ((3 * P + 12) * 8 + 4)

    if rank != 0:
        return 0
    # dominant kernel and its roofline: algorithmic FP64 flops per launch over
    # the launch's CUDA-event duration, against the measured FP64 FMA rate
    dom = max((k for k in kt if kt[k][1] > 0), key=lambda k: kt[k][0])
    share = {k: round(kt[k][0] / max(1e-12, sum(v[0] for v in kt.values())), 4) for k in kt}
    from paper_2602_13553_gb300 import inputs
    rc = inputs.WATER_FF[6]
    overhead = None
    if dom == "force":
        flops, overhead = force_flops(xs, w["L"], rc, rc + 1.5)
        kname = "k_force_water_f64"
    else:
        flops = step_flops_per_bead_atom(P) * N * P
        kname = "k_step_f64" if dom == "step" else dom
    avg_ms = kt[dom][0] / kt[dom][1]
    achieved = flops / (avg_ms / 1e3) / 1e12
    md_ms = total_ms / args.steps / w["md_per_step"]
    hbm, hsrc = hbm_peak()
    line = {
        "metric": METRIC, "value": value, "unit": METRIC, "n_gpus": world, "steps": args.steps,
        "warmup": max(3, args.warmup), "ms_per_step": total_ms / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": config({"parallelism": "replicas" if world > 1 else "single",
                                               "md_step_latency_us": md_ms * 1e3}),
        "roofline": {"bound": "alu", "kernel": kname, "achieved": achieved, "peak": fp64_peak,
                     "unit": "TFLOP/s", "frac": achieved / fp64_peak,
                     "peak_source": "measured: FP64 FMA throughput of this GPU (pimd_fp64_fma_rate), "
                                    "nominal %.2f" % (FP64_NOMINAL / 1e12),
                     "algorithmic_flops_per_launch": flops,
                     "overhead_flops_per_launch": overhead,
                     "avg_launch_ms": avg_ms, "kernel_time_share": share,
                     "note": "the 0.44 MB state stays in L2: a latency-bound workload whose "
                             "figure of merit is the %.1f us per MD step" % (md_ms * 1e3),
                     "hbm": {"achieved": 168.0 * N * P / (md_ms / 1e3) / 1e9, "peak": hbm,
                             "unit": "GB/s", "peak_source": hsrc,
                             "basis": "168 B per bead-atom-step (step 120 + force 48) over the "
                                      "whole MD step"}},
        "e2e": {"value": e2e_value, "unit": METRIC, "h2d_bytes_per_step": h2d,
                "d2h_bytes_per_step": d2h,
                "path": "pimd_set_state (pinned host x, v) + 10 x (pimd_step(100) + pimd_estimators)"},
        "gpu_launches": int(launches),
        "clocks": clk,
    }
    if world == 1 and not args.no_batched:
        line["batched"] = batched_bench(stream, args.batched_steps, 3)
        line["batched"]["vs_plain_fp64"] = line["batched"]["value"] / value
    if world == 1 and not args.no_serve:
        line["serve"] = serve_bench(stream, args.serve_jobs, args.serve_step_scale)
    if world == 1 and not args.no_sweep:
        line["sweep"] = sweep_bench(stream)
    if not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline()
        line["cpu_baseline"]["configs"] = oracle_configs()
    print(json.dumps(line))
    sim.close()
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
