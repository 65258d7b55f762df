"""Benchmark of the electrokinetic LB-MD step on GB300.

Workload (default): the 256 x 256 x 512 translocation pore (33.5 M D3Q19
nodes), membrane 16 thick centred at z = 256, cylindrical pore of radius 8,
1:1 salt 0.01, E_z = 2e-3, a 128-bead FENE+WCA chain threaded through the
pore, FP32 populations, Poisson by multigrid-preconditioned CG to relative
residual 1e-8.  A step is one whole time step (charge, Poisson, beads, fused
LB update).  The 64 x 64 x 128 pore (radius 4, N = 32, salt 0.005,
E_z = 5e-3) is measured beside it under the key "pore_64x64x128".

Metric: species-MLUPS = lattice nodes x 3 species x steps / s / 1e6, plus
steps/s; the dominant kernel and the fused LB kernel are reported against
the HBM roofline.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Under torchrun (N > 1) every rank runs its own independent replica (the path
has no data exchange between replicas), timing is the max over ranks and the
value is the aggregate over all ranks.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "EK-LB-MD steps/s & species-MLUPS vs HBM roofline; learned vs plain Poisson"
UNIT = "species-MLUPS"
FALLBACK_HBM_GBS = 6800.0

# DRAM bytes per launch from the committed ncu captures (profiles/<kernel>_<workload>.md),
# keyed by kernel and workload, each valid only while the source files it was
# taken on are unchanged
PROFILED = {
    # (kernel, workload): (sha256 prefix of its source files, dram read + write bytes per launch), from one
    # ncu pass over the benchmark command (--graph-profiling graph; the split solve's figure is its start
    # kernel plus its graph, the mean over the capture's solves: 6.4 CG iterations on 256x256x512, 5.2 on
    # 64x64x128)
    ("lb_fused_kernel", "pore_256x256x512_r8_N128"): ("10a11f244e6a891f", 7824038613 + 7365457280),
    ("multigrid_split_solve", "pore_256x256x512_r8_N128"): ("709bbd944d326a48",
                                                         674914076 + 696878222 + 20891236423 + 7463117483),
    ("lb_fused_kernel", "pore_64x64x128_r4_N32"): ("10a11f244e6a891f", 119390228 + 63359449),
    ("multigrid_split_solve", "pore_64x64x128_r4_N32"): ("709bbd944d326a48", 10722934 + 0 + 17523436 + 45076),
}
KERNEL_SOURCES = {
    "lb_fused_kernel": ("ekl_kernels.cuh", "ekl_dev.cuh"),
    "poisson_mg_kernel": ("ekl_mg.cuh", "ekl_kernels.cuh", "ekl_dev.cuh"),
    "poisson_mg_wide_kernel": ("ekl_mg.cuh", "ekl_kernels.cuh", "ekl_dev.cuh"),
    "multigrid_split_solve": ("ekl_mgs.cuh", "ekl_mgf.cuh", "ekl_mg.cuh", "ekl_kernels.cuh", "ekl_dev.cuh"),
    "poisson_tiled_kernel": ("ekl_kernels.cuh", "ekl_rim.h", "ekl_dev.cuh"),
}


def n_sms():
    try:
        import torch
        return torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count
    except Exception:
        return 152


def source_sha16(kernel):
    import hashlib
    h = hashlib.sha256()
    for f in KERNEL_SOURCES.get(kernel, ()):
        h.update(open(os.path.join(ROOT, "paper_1710_09421_gb300", "csrc", f), "rb").read())
    return h.hexdigest()[:16]


def profiled_traffic(kernel, workload):
    sha, traffic = PROFILED.get((kernel, workload), (None, None))
    return traffic if sha is not None and sha == source_sha16(kernel) else None


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return FALLBACK_HBM_GBS, "fallback"


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""

    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index=0):
        self.index = index
        self.rows = []
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
            time.sleep(0.3)
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 7:
                self.rows.append(parts)

    def __exit__(self, *a):
        if self.proc:
            time.sleep(0.2)
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        if not self.rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        sm = [float(r[0]) for r in self.rows if r[0].replace(".", "").isdigit()]
        mx = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in self.rows for k in range(4) if r[3 + k] == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(self.rows)}


def poisson_algorithmic_bytes(wl, sweeps):
    """Bytes a streamed red-black SOR would move for `sweeps` sweeps: per
    fluid node and sweep the source (8 B), the link word (4 B), its own
    potential read and written (8 + 8 B); the neighbours come from cache."""
    nf = int((wl.solid == 0).sum())
    return sweeps * nf * 28


# Multigrid solve, per fluid node (FP32 path, 8-byte fixed-point potential),
# with L bytes of link data per node (the split solve reads a 1-byte link
# array, the single cooperative launch the 4-byte link word): per CG
# iteration 5.5 lattice sweeps x (12 + L) B (r, z read, z written, link),
# restriction 8 + L, p/q pass 16 + L, update pass 34 + L, coarse levels 14 B
# (1/7 of the lattice smoothing and restriction); per solve the source
# (12 + L) and two true-residual passes (22 + L each).
def mg_bytes_per_iter(L):
    return 5.5 * (12 + L) + (8 + L) + (16 + L) + (34 + L) + 14


def mg_bytes_per_solve(L):
    return (12 + L) + 2 * (22 + L)


# The same where the split solve takes two half sweeps per launch (1-byte link
# array): r (4 B) and the link byte in every pass, and the colour-0 values
# between passes, 2 B a node: pre-smoothing 5 + 2 written; restriction 5 + 2,
# and the coarse right-hand side and first values 1; prolongation 5 + 2 + 2 and
# the coarse correction 0.5; last pass 5 + 2 and z written 4; r.z 9; p/q pass 17;
# update pass 33 (it no longer starts z); coarse levels 14.  The first residual no
# longer starts z either.
MG_FUSED_BYTES_PER_ITER = 7 + 8 + 9.5 + 11 + 9 + 17 + 33 + 14
MG_FUSED_BYTES_PER_SOLVE = 13 + 21 + 23


MG_SPLIT_KERNELS_PER_SOLVE = 5  # start, first true residual, init, final residual, report


def mg_split(W, wl, sms=152):
    return bool(wl.flags & W.FLAG_POISSON_MG) and not (wl.flags & W.FLAG_POISSON_MG_SINGLE)


def mg_fused(W, wl, sms=152):
    """Two half sweeps per launch: lattices whose solve (37 B a node) does not
    stay in 126 MB of L2, in 1024-thread blocks, with rows of whole groups of four."""
    return (mg_split(W, wl, sms) and wl.nx % 4 == 0 and wl.n_nodes >= 16384 * sms
            and wl.n_nodes * 37 > 126 << 20)


def mg_split_kernels_per_iter(wl, sms=152, fused=False):
    """Launches per CG iteration of the split solve: 14, or 11 with two half
    sweeps per launch, plus 8 when level 1 is too large for shared-memory tiles
    (more than 1024 cells per block)."""
    level1 = ((wl.nx + 1) // 2) * ((wl.ny + 1) // 2) * ((wl.nz + 1) // 2)
    return (11 if fused else 14) + (8 if level1 > 1024 * sms else 0)


def mg_algorithmic_bytes(wl, iters, link_bytes=4, fused=False):
    nf = int((wl.solid == 0).sum())
    if fused:
        return nf * (iters * MG_FUSED_BYTES_PER_ITER + MG_FUSED_BYTES_PER_SOLVE)
    return nf * (iters * mg_bytes_per_iter(link_bytes) + mg_bytes_per_solve(link_bytes))


def lb_algorithmic_bytes(wl, store_bytes):
    """Bytes one fused-LB launch must move at minimum: per fluid node 57
    populations read and written, the link word and the potential (8 B, the
    6 neighbours come from cache); per wall node the link word."""
    nf = int((wl.solid == 0).sum())
    ns = wl.n_nodes - nf
    return nf * (2 * 57 * store_bytes + 4 + 8) + ns * 4


def dist_setup(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        backend = "nccl" if args.impl == "ours" else "gloo"
        dist.init_process_group(backend=backend)
    return world, rank, local


def max_over_ranks(x, world):
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64,
                     device="cuda" if dist.get_backend() == "nccl" else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def workload_for(name, rank=0, args=None):
    from paper_1710_09421_gb300 import workloads as W
    if name == "pore3":
        wl = W.config_precision_sweep("f32")
    elif name == "pore5":
        wl = W.config_learned("f32")
    elif name == "pore":
        wl = W.config_pore_fp32()
    elif name == "slit":
        wl = W.config_slit_fp64().replace(precision="f32", poisson_tol=1e-8)
    else:
        raise SystemExit(f"unknown workload {name}")
    if rank:
        wl = wl.replace(seed=wl.seed + 1000 * rank)  # independent replica per rank
    if args is not None and args.rho_jacobi > 0:
        wl = wl.replace(rho_jacobi=args.rho_jacobi)
    if args is not None and args.check_every > 0:
        wl = wl.replace(poisson_check_every=args.check_every)
    if args is not None and getattr(args, "poisson", "sor") == "mg":
        wl = wl.replace(flags=wl.flags | W.FLAG_POISSON_MG)
    return wl


# The oracle's Chebyshev SOR needs thousands of sweeps per step on lattices of
# tens of millions of nodes (minutes per step); its bounded sample there runs
# whole steps with the solve cut to this many sweeps.
SAMPLE_SWEEPS = 10
ORACLE_FULL_SOLVE_NODES = 1 << 21
# host bytes the oracle holds per lattice node (FP64 populations 2 x 57 x 8,
# moments, bead forces, potential, source, gradient, wall map)
ORACLE_BYTES_PER_NODE = 1200


def host_mem_available():
    try:
        for line in open("/proc/meminfo"):
            if line.startswith("MemAvailable:"):
                return int(line.split()[1]) * 1024
    except OSError:
        pass
    return 0


def oracle_sample(wl, threads, budget_s, max_steps=50, warm=True):
    """The oracle, as it stands, timed over whole steps of wl (a bounded
    sample: at most max_steps steps or budget_s seconds).  Lattices above
    ORACLE_FULL_SOLVE_NODES run with the Poisson solve cut to SAMPLE_SWEEPS
    sweeps.  Returns (species-MLUPS, steps, seconds, truncated)."""
    import oracle
    trunc = wl.n_nodes > ORACLE_FULL_SOLVE_NODES
    ref = oracle.Sim(wl.replace(poisson_fixed_iter=SAMPLE_SWEEPS) if trunc else wl, threads=threads)
    if warm:
        ref.step(1)  # the first step of a full solve starts cold
    t0 = time.perf_counter()
    n = 0
    while True:
        ref.step(1)
        n += 1
        if time.perf_counter() - t0 > budget_s or n >= max_steps:
            break
    dt = time.perf_counter() - t0
    del ref
    return wl.n_nodes * 3 * n / dt / 1e6, n, dt, trunc


def cpu_baseline(wl, small_wl, budget_s=20.0):
    """The oracle on the host cores: all cores on a bounded sample of the
    benchmarked workload (whole steps; the Poisson solve cut to SAMPLE_SWEEPS
    sweeps on lattices too large for its full solve, which overstates the
    oracle's rate), and all cores and one thread on the 64 x 64 x 128 pore
    with its full solve.  Values in species-MLUPS."""
    cores = os.cpu_count() or 1
    out = {"unit": UNIT, "cores": cores, "kind": "oracle"}
    if wl.n_nodes * ORACLE_BYTES_PER_NODE * 1.5 < host_mem_available():
        v, n, dt, trunc = oracle_sample(wl, cores, budget_s, warm=not wl.n_nodes > ORACLE_FULL_SOLVE_NODES)
        out["value"] = round(v, 4)
        out["sample"] = (f"{n} oracle step(s) of the whole {wl.name} lattice, FP64, {cores} threads, "
                         f"{dt:.1f} s" + (f"; Chebyshev SOR cut to {SAMPLE_SWEEPS} sweeps per step (the "
                                          "full solve needs thousands here), so this overstates the "
                                          "oracle's rate" if trunc else ""))
    else:
        out["value"] = None
        out["sample"] = f"skipped: the oracle needs {wl.n_nodes * ORACLE_BYTES_PER_NODE / 1e9:.0f} GB of host memory"
    v, n, dt, _ = oracle_sample(small_wl, cores, budget_s / 4, max_steps=5)
    out[small_wl.name] = {"value": round(v, 4), "threads": cores,
                          "sample": f"{n} full oracle steps after 1 warm-up step, {dt:.1f} s"}
    import oracle
    ref = oracle.Sim(small_wl, threads=cores)
    ref.step(1)
    ref.set_threads(1)
    t0 = time.perf_counter()
    ref.step(1)
    dt = time.perf_counter() - t0
    out["single_thread"] = {"value": round(small_wl.n_nodes * 3 / dt / 1e6, 4), "threads": 1,
                            "sample": f"1 full oracle step of the {small_wl.name} workload after 1 "
                                      f"warm-up step, {dt:.1f} s"}
    if out["value"] is None:
        out["value"] = out[small_wl.name]["value"]
        out["sample"] += f"; value is the {small_wl.name} sample"
    return out


def run_batch(args):
    """Batched replicas (one launch per phase for all replicas): aggregate
    species-MLUPS and translocation events per hour."""
    import numpy as np
    import torch

    import paper_1710_09421_gb300 as E
    from paper_1710_09421_gb300 import workloads as W

    torch.cuda.set_device(0)
    E.load()
    wls = W.replica_set(n_rep=args.replicas, precision=args.precision)
    if args.poisson == "mg":
        wls = [w.replace(flags=w.flags | W.FLAG_POISSON_MG) for w in wls]
    stream = torch.cuda.Stream()
    b = E.Batch(wls, stream=stream.cuda_stream)
    choice = b.autotune(1)
    for _ in range(args.warmup):
        b.step(1)
    z_mid = [0.5 * (w.nz - 1) for w in wls]
    l0 = b.launches()
    torch.cuda.synchronize()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    with ClockSampler(0) as clk:
        ev0.record(stream)
        rc = b.step(args.steps)
        ev1.record(stream)
        torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1)
    launches = b.launches() - l0
    nodes = sum(w.n_nodes for w in wls)
    steps_per_s = args.steps / (ms / 1e3)
    # translocation events: every bead of a chain past its pore's midplane
    # along the field (-z for negative beads), counted at the end of the run
    events = 0
    for r, w in enumerate(wls):
        if not w.n_beads:
            continue
        z = b.reps[r].fields(("R",))["R"][:, 2]
        if np.all(z < z_mid[r]):
            events += 1
    sweeps = np.mean([b.reps[r].stats()["poisson_iters"] for r in range(len(wls))])
    line = {
        "metric": METRIC, "value": round(nodes * 3 * steps_per_s / 1e6, 3), "unit": UNIT, "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms / args.steps, 3),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": args.precision,
        "data": "synthetic",
        "config": {"workload": f"{len(wls)} uneven translocation replicas", "nodes": nodes,
                   "beads": int(sum(w.n_beads for w in wls)), "poisson_tol": wls[0].poisson_tol,
                   "autotune_choice": choice, "l2": "inputs larger than L2"},
        "poisson_solver": "multigrid-CG" if args.poisson == "mg" else "chebyshev-sor",
        "steps_per_s": round(steps_per_s, 3), "poisson_iterations_last_step_mean": float(sweeps),
        "events_completed": events,
        "events_note": "counted over the %d timed steps; at this rate a chain of 16 beads needs about 10^4 "
                       "steps to translocate, so short runs complete none" % args.steps,
        "gpu_launches": launches, "clocks": clk.summary(), "status": rc,
    }
    print(json.dumps(line))
    b.close()


def run_precision(args):
    """Storage-precision sweep on the 256x256x512 pore (membrane 16 thick,
    radius 8, N = 128): the same run in FP64 and in FP32 / BF16 / FP16
    deviation storage (FP32 arithmetic), errors against the FP64 run per
    observable, and each format's throughput."""
    import numpy as np
    import torch

    import paper_1710_09421_gb300 as E
    from paper_1710_09421_gb300 import workloads as W

    torch.cuda.set_device(0)
    E.load()
    base = W.config_precision_sweep()
    if args.poisson == "mg":
        base = base.replace(flags=base.flags | W.FLAG_POISSON_MG)
    fluid = base.solid.ravel() == 0
    every = max(1, min(10, args.steps // 100))
    out = {}
    ref = None
    for prec in ("f64", "f32", "bf16", "fp16"):
        sim = E.Simulation(base, precision=prec)
        zs = []
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for k in range(0, args.steps, every):
            sim.step(min(every, args.steps - k))
            zs.append(float(sim.fields(("R",))["R"][:, 2].mean()))
        torch.cuda.synchronize()
        dt = time.perf_counter() - t0
        F = sim.fields(("n", "j", "phi"))
        st = sim.stats()
        sim.close()
        u = F["j"] / np.where(F["n"] > 0, F["n"], 1.0)[:, None, :]
        rec = {"steps_per_s": round(args.steps / dt, 3), "poisson_iters_last": st["poisson_iters"],
               "status": st["status"]}
        if ref is None:
            ref = (F, u, np.array(zs))
        else:
            F0, u0, z0 = ref
            scale = max(np.linalg.norm(u0[a][:, fluid]) for a in range(3))
            rec["err_n_ions"] = float(max(np.linalg.norm(F["n"][a][fluid] - F0["n"][a][fluid]) /
                                          np.linalg.norm(F0["n"][a][fluid]) for a in (1, 2)))
            rec["err_u_flow"] = float(max(np.linalg.norm(u[a][:, fluid] - u0[a][:, fluid]) / scale
                                          for a in range(3)))
            rec["err_phi"] = float(np.linalg.norm(F["phi"][fluid] - F0["phi"][fluid]) /
                                   np.linalg.norm(F0["phi"][fluid]))
            dz = np.array(zs) - z0
            rec["err_bead_z_max"] = float(np.abs(dz).max())
            rec["bead_z_drift_f64"] = float(z0[-1] - z0[0])
        # translocation progress: the step at which the chain's centre of mass
        # has moved CROSS_DZ lattice units along the field (interpolated)
        rec["progress_step"] = progress_step(zs, every)
        if prec != "f64" and out["f64"]["progress_step"] is not None and rec["progress_step"] is not None:
            rec["err_progress_steps"] = round(rec["progress_step"] - out["f64"]["progress_step"], 2)
        out[prec] = rec
        del F, u
    line = {"metric": "storage-precision error vs the FP64 run", "unit": "relative / lattice units / steps",
            "progress_definition": "step at which the chain's mean z has moved %.1f lattice units along the field"
                                   % CROSS_DZ,
            "steps": args.steps, "config": {"workload": base.name, "nodes": base.n_nodes, "beads": base.n_beads,
                                            "poisson_tol": base.poisson_tol},
            "data": "synthetic", "precisions": out}
    print(json.dumps(line))


CROSS_DZ = 2.0


def progress_step(zs, every, dz=CROSS_DZ):
    """First step at which the recorded mean bead z (sampled every `every`
    steps, zs[0] after the first sample interval) lies dz below the first
    sample, by linear interpolation between samples; None if never."""
    z0 = zs[0]
    for k in range(1, len(zs)):
        if zs[k] <= z0 - dz:
            a, b = zs[k - 1] - (z0 - dz), zs[k - 1] - zs[k]
            return round(every * (k + (a / b if b else 1.0)), 2)
    return None


def run_reference(args):
    """The oracle (the only reference implementation: the paper ships no
    code) on the benchmarked workload, each step a bounded sample (whole steps
    of the whole lattice; on lattices too large for its full solve the
    Chebyshev SOR is cut to SAMPLE_SWEEPS sweeps per step)."""
    world, rank, local = dist_setup(args)
    if rank != 0:
        return
    wl = workload_for(args.workload, 0, args)
    cores = os.cpu_count() or 1
    if wl.n_nodes * ORACLE_BYTES_PER_NODE * 1.5 >= host_mem_available():
        print(json.dumps({"impl": "reference", "unavailable":
                          f"the oracle needs {wl.n_nodes * ORACLE_BYTES_PER_NODE / 1e9:.0f} GB of host "
                          "memory for this lattice"}))
        return
    budget = 90.0
    value, n, dt, trunc = oracle_sample(wl, cores, budget, max_steps=args.steps, warm=True)
    solver = "chebyshev-sor" + (f" cut to {SAMPLE_SWEEPS} sweeps per step" if trunc else f" to {wl.poisson_tol:g}")
    line = {
        "impl": "reference", "metric": METRIC, "value": round(value, 4), "unit": UNIT,
        "n_gpus": args.gpus, "steps": n, "warmup": 1,
        "ms_per_step": round(1e3 * dt / n, 3), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": wl.name, "nodes": wl.n_nodes, "species": 3, "beads": wl.n_beads,
                   "poisson_tol": wl.poisson_tol, "poisson_solver": solver,
                   "note": "the FP64 CPU oracle; its Poisson solver is the paper's Chebyshev SOR, "
                           "the GPU arm's is multigrid-CG to the same residual"},
        "cpu_baseline": {"value": round(value, 4), "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": f"{n} of {args.steps} requested steps (time-capped at {budget:.0f} s) "
                                   f"on the whole lattice after 1 warm-up step; Poisson: {solver}"},
        "e2e": {"value": round(value, 4), "unit": UNIT, "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))


def measure(E, W, wl, args, sraw, local, world, phase_steps):
    """Warm-up, then exactly args.steps timed steps with CUDA events on the
    library's stream (no per-phase events inside), then a separate window of
    phase_steps steps with per-phase events for the phase times and the
    per-kernel rooflines."""
    import torch

    sim = E.Simulation(wl, precision=args.precision, stream=sraw)
    for _ in range(args.warmup):
        sim.step(1)
    st0 = sim.stats()
    barrier(world)
    torch.cuda.synchronize()
    stream = torch.cuda.ExternalStream(sraw)
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clk:
        ev0.record(stream)
        rc = sim.step(args.steps)
        ev1.record(stream)
        torch.cuda.synchronize()
    barrier(world)
    ms = ev0.elapsed_time(ev1)
    st1 = sim.stats()
    sim.set_timing(True)
    sim.step(phase_steps)
    st2 = sim.stats()
    sim.close()
    return dict(ms=ms, rc=rc, clocks=clk.summary(), launches=st1["launches"] - st0["launches"],
                iters=(st1["poisson_sweeps"] - st0["poisson_sweeps"]) / args.steps,
                phase={k: v / phase_steps for k, v in st2["ms_phase"].items()},
                phase_iters=(st2["poisson_sweeps"] - st1["poisson_sweeps"]) / phase_steps,
                res=st1["poisson_res"])


def rooflines(W, wl, m, store):
    """Roofline objects of the Poisson solve and of the fused LB kernel from
    the phase window of measure()."""
    hbm, peak_kind = peaks()
    mg = bool(wl.flags & W.FLAG_POISSON_MG)
    ph = m["phase"]
    split = mg and mg_split(W, wl, n_sms())
    fused = split and mg_fused(W, wl, n_sms())
    if split:
        pk = "multigrid_split_solve"
        pb = mg_algorithmic_bytes(wl, m["phase_iters"], link_bytes=1, fused=fused)
    elif mg:
        pk = "poisson_mg_wide_kernel" if wl.n_nodes >= 152 * 16384 else "poisson_mg_kernel"
        pb = mg_algorithmic_bytes(wl, m["phase_iters"])
    else:
        pk = "poisson_tiled_kernel" if wl.n_nodes <= 1 << 21 else "poisson_kernel"
        pb = poisson_algorithmic_bytes(wl, m["phase_iters"])
    pa = pb / (ph["poisson"] / 1e3) / 1e9
    lb = lb_algorithmic_bytes(wl, store)
    la = lb / (ph["lb"] / 1e3) / 1e9
    pois = {"kernel": pk, "bound": "hbm", "achieved": round(pa, 1), "peak": hbm, "unit": "GB/s",
            "frac": round(pa / hbm, 4), "peak_kind": peak_kind, "traffic": profiled_traffic(pk, wl.name),
            "algorithmic_bytes_per_launch": int(pb), "avg_launch_ms": round(ph["poisson"], 5)}
    if split and pois["traffic"] is not None:
        pois["traffic_note"] = ("ncu, one pass: the start kernel plus the solve's graph, mean over the capture's "
                                "solves (6.4 CG iterations on 256x256x512, 5.2 on 64x64x128)")
    if split:
        pois["launches_per_solve"] = round(MG_SPLIT_KERNELS_PER_SOLVE + mg_split_kernels_per_iter(wl, n_sms(), fused)
                                           * m["phase_iters"], 1)
        pois["unit_measured"] = ("the whole solve, timed with CUDA events on its stream: a start kernel and one graph "
                                 "launch (lattice passes " + ("two half sweeps" if fused else "one half sweep") +
                                 " per kernel, the coarse levels of each V-cycle one "
                                 "cooperative kernel, the CG loop a conditional WHILE node); bytes and time per solve")
    lbr = {"kernel": "lb_fused_kernel", "bound": "hbm", "achieved": round(la, 1), "peak": hbm,
           "unit": "GB/s", "frac": round(la / hbm, 4), "peak_kind": peak_kind,
           "traffic": profiled_traffic("lb_fused_kernel", wl.name),
           "algorithmic_bytes_per_launch": lb, "avg_launch_ms": round(ph["lb"], 5)}
    return pois, lbr


def run_ours(args):
    world, rank, local = dist_setup(args)
    import torch

    torch.cuda.set_device(local)
    import paper_1710_09421_gb300 as E
    from paper_1710_09421_gb300 import workloads as W

    E.load()
    wl = workload_for(args.workload, rank, args)
    stream = torch.cuda.Stream()
    sraw = stream.cuda_stream
    store = {"f32": 4, "f64": 8, "bf16": 2, "fp16": 2}[args.precision]
    phase_steps = max(5, min(args.steps, 20))

    # ---- device-resident timed run
    m = measure(E, W, wl, args, sraw, local, world, phase_steps)
    ms_max = max_over_ranks(m["ms"], world)
    value = wl.n_nodes * args.steps * world * 3 / (ms_max / 1e3) / 1e6
    steps_per_s = args.steps * world / (ms_max / 1e3)
    pois_roof, lb_roof = rooflines(W, wl, m, store)
    dominant = max(("poisson", "lb", "charge", "bead_md", "bead_bin"), key=lambda k: m["phase"][k])
    share = f"{100 * m['phase'][dominant] / sum(m['phase'].values()):.0f} %"
    if pois_roof["kernel"] == "multigrid_split_solve":
        pois_roof["note"] = (f"dominant phase ({dominant}: {share} of the phase times), measured as one unit; "
                             "its kernels' shares are in the ncu launch list")
    else:
        pois_roof["note"] = f"dominant kernel ({dominant} phase: {share} of the phase times); one launch = one step's solve"

    # ---- end to end through the public API: host inputs in, fields out
    torch.cuda.synchronize()
    barrier(world)
    t0 = time.perf_counter()
    sim2 = E.Simulation(wl, precision=args.precision, stream=sraw)
    sim2.step(args.steps)
    F = sim2.fields(("n", "j", "phi", "R", "V"))
    torch.cuda.synchronize()
    t1 = time.perf_counter()
    sim2.close()
    del F
    e2e_s = max_over_ranks(t1 - t0, world)
    h2d = wl.n_nodes * (1 + 3 * 8) + (wl.n_beads * (3 + 3 + 1) * 8)
    if wl.surface_charge is not None:
        h2d += wl.n_nodes * 8
    d2h = wl.n_nodes * (3 + 9 + 1) * 8 + wl.n_beads * 6 * 8
    e2e_val = wl.n_nodes * args.steps * world * 3 / e2e_s / 1e6

    # ---- the 64 x 64 x 128 pore beside it
    small = None
    if args.workload != "pore":
        swl = workload_for("pore", rank, args)
        ms_ = measure(E, W, swl, args, sraw, local, world, phase_steps)
        sp, sl = rooflines(W, swl, ms_, store)
        small = {"workload": swl.name, "nodes": swl.n_nodes,
                 "value": round(swl.n_nodes * args.steps * 3 / (ms_["ms"] / 1e3) / 1e6, 3),
                 "steps_per_s": round(args.steps / (ms_["ms"] / 1e3), 3),
                 "ms_per_step": round(ms_["ms"] / args.steps, 4),
                 "poisson_iterations_per_step": round(ms_["iters"], 2),
                 "phase_ms_per_step": {k: round(v, 5) for k, v in ms_["phase"].items()},
                 "roofline": sp, "roofline_lb": sl, "clocks": ms_["clocks"], "status": ms_["rc"]}

    if rank != 0:
        return
    mg = bool(wl.flags & W.FLAG_POISSON_MG)
    line = {
        "metric": METRIC, "value": round(value, 3), "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms_max / args.steps, 4),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": {"f32": "f32", "f64": "f64", "bf16": "bf16-storage/f32", "fp16": "fp16-storage/f32"}[args.precision],
        "data": "synthetic",
        "config": {"workload": wl.name, "nodes": wl.n_nodes, "species": 3, "beads": wl.n_beads,
                   "precision": args.precision, "poisson_tol": wl.poisson_tol,
                   "l2": "inputs larger than L2 (populations 2 x %.0f MB)" % (
                       wl.n_nodes * 57 * store / 1e6)},
        "steps_per_s": round(steps_per_s, 3),
        "poisson_solver": "multigrid-CG" if mg else "chebyshev-sor",
        "poisson_iterations_per_step": round(m["iters"], 2),
        "poisson_res_last": m["res"],
        "phase_ms_per_step": {k: round(v, 5) for k, v in m["phase"].items()},
        "phase_window": f"{phase_steps} steps after the timed region, per-phase CUDA events",
        "roofline": pois_roof,
        "roofline_lb": lb_roof,
        "clocks": m["clocks"],
        "gpu_launches": m["launches"],
        "e2e": {"value": round(e2e_val, 3), "unit": UNIT,
                "h2d_bytes_per_step": int(h2d / args.steps), "d2h_bytes_per_step": int(d2h / args.steps),
                "what": "create from host arrays + beads + %d steps + all fields to host" % args.steps},
        "status": m["rc"],
    }
    if small is not None:
        line["pore_64x64x128"] = small
    if world == 1 and not args.no_learned:
        line["learned_vs_plain"] = learned_summary(E, W, args, sraw)
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(wl, workload_for("pore", 0, args), budget_s=args.cpu_budget)
    print(json.dumps(line))


def learned_vs_plain(E, wl, args, sraw, collect_steps=60, ncrops=8, crop=16, train_iters=400,
                     compare_steps=40, train_wl=None, trained=None, level=0):
    """Train the warm-start network on samples the solver records on train_wl
    (default: this workload; a separate run with another seed), or take a
    trained (weights, scales, info), then time the same steps with and
    without it from identical states.  Both runs iterate to the same
    residual tolerance; only sweeps and time are compared.  level: the
    lattice level the network runs on (0: the lattice, crops near the beads;
    L >= 1: whole grids of 2^L-node cells)."""
    import torch

    if trained is None:
        trained = train_warmstart(E, train_wl or wl, args, sraw, collect_steps, ncrops, crop, train_iters, level)
    w, scales, info = trained
    out = dict(info)
    for name, use in (("plain", False), ("learned", True)):
        sim = E.Simulation(wl, precision=args.precision, stream=sraw)
        sim.step(args.warmup)
        if use:
            sim.set_warmstart(w, scales, level=level)
        sim.step(2)   # the network needs the previous source
        s0 = sim.stats()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        st = torch.cuda.ExternalStream(sraw) if sraw else torch.cuda.current_stream()
        e0.record(st)
        sim.step(compare_steps)
        e1.record(st)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1)
        s1 = sim.stats()
        sim.close()
        out[name] = {"steps_per_s": round(compare_steps / (ms / 1e3), 3),
                     "poisson_sweeps_per_step": round((s1["poisson_sweeps"] - s0["poisson_sweeps"]) / compare_steps, 2),
                     "poisson_res_last": s1["poisson_res"]}
    out["sweeps_saved_frac"] = round(1 - out["learned"]["poisson_sweeps_per_step"]
                                     / max(out["plain"]["poisson_sweeps_per_step"], 1e-9), 4)
    out["speedup"] = round(out["learned"]["steps_per_s"] / max(out["plain"]["steps_per_s"], 1e-9), 4)
    return out


def train_warmstart(E, wl, args, sraw, collect_steps, ncrops, crop, train_iters, level=0):
    """Samples recorded by the solver on wl with another seed, and the
    network trained on them: (weights, scales, info)."""
    import numpy as np
    from paper_1710_09421_gb300 import warmstart as WS

    t0 = time.perf_counter()
    src = E.Simulation(wl.replace(seed=wl.seed + 101), precision=args.precision, stream=sraw)
    src.step(args.warmup)
    if level:
        src.warmstart_level(level)
        data = src.collect(collect_steps + 1, seed=7)[1:]  # the first step has no previous source
    else:
        data = src.collect(collect_steps, crop=crop, ncrops=ncrops, seed=7)
    src.close()
    t1 = time.perf_counter()
    if level:
        w, scales, curve = WS.train_fields(data, wl.periodic, iters=train_iters, batch=8, lr=2e-3, seed=0)
    else:
        w, scales, curve = WS.train(data, iters=train_iters, batch=8, lr=2e-3, seed=0)
    t2 = time.perf_counter()
    info = {"samples": int(len(data)), "level": level, "collect_s": round(t1 - t0, 3),
            "train_s": round(t2 - t1, 3), "train_iters": train_iters,
            "rel_loss_first": round(float(np.mean(curve[:20])), 4),
            "rel_loss_last": round(float(np.mean(curve[-20:])), 4)}
    if not level:
        info["crop"] = crop
    return w, scales, info


def learned_summary(E, W, args, sraw, samples=2000, iters=600):
    """The learned warm start in the benchmark line: trained on the
    64x64x128 pore (another seed) at network level --ws-level, compared on
    the 128x128x256 pore with the paper's SOR and with multigrid, at the same
    residual (the full-size training of BASELINE's 20 000 snapshots is
    `--workload learned`)."""
    wl = W.config_learned(args.precision)
    train_wl = W.config_pore_fp32().replace(flags=W.FLAG_POISSON_MG)
    L = args.ws_level
    trained = train_warmstart(E, train_wl, args, sraw, collect_steps=samples, ncrops=1, crop=0,
                              train_iters=iters, level=L)
    out = {"workload": "pore_128x128x256_r6_N64", "trained_on": "pore_64x64x128_r4_N32, seed + 101",
           "network_level": L}
    sor = wl.replace(rho_jacobi=0.9999, poisson_check_every=4, poisson_max_iter=20000)
    for name, w_ in (("chebyshev-sor", sor), ("multigrid-CG", wl.replace(flags=wl.flags | W.FLAG_POISSON_MG))):
        r = learned_vs_plain(E, w_, args, sraw, compare_steps=12, trained=trained, level=L)
        out[name] = {k: r[k] for k in ("plain", "learned", "sweeps_saved_frac", "speedup")}
        out["training"] = {k: r[k] for k in ("samples", "train_iters", "rel_loss_first", "rel_loss_last",
                                             "collect_s", "train_s")}
    return out


def run_learned(args):
    """The learned warm start on the 128x128x256 pore (radius 6, N = 64,
    salt 0.005): the network is trained on samples that the solver records
    on the 64x64x128 pore (radius 4, N = 32) under another seed, then the
    same steps run with and without it from identical states, to the same
    residual, with the paper's Chebyshev SOR and with multigrid.  The
    network runs on cells of 2^level nodes (--ws-level)."""
    import torch

    import paper_1710_09421_gb300 as E
    from paper_1710_09421_gb300 import workloads as W

    torch.cuda.set_device(0)
    E.load()
    stream = torch.cuda.Stream()
    sraw = stream.cuda_stream
    wl = W.config_learned(args.precision)
    train_wl = W.config_pore_fp32().replace(flags=W.FLAG_POISSON_MG)
    L = args.ws_level
    if L:
        trained = train_warmstart(E, train_wl, args, sraw, collect_steps=args.ws_samples, ncrops=1, crop=0,
                                  train_iters=args.ws_iters, level=L)
    else:
        trained = train_warmstart(E, train_wl, args, sraw, collect_steps=250, ncrops=80, crop=16,
                                  train_iters=800)
    line = {"metric": "learned vs plain Poisson: iterations and steps/s at the same residual",
            "unit": "steps/s", "data": "synthetic", "dtype": args.precision,
            "config": {"workload": "pore_128x128x256_r6_N64", "nodes": wl.n_nodes,
                       "poisson_tol": wl.poisson_tol, "trained_on": "pore_64x64x128_r4_N32, seed + 101",
                       "network_level": L}}
    sor = wl.replace(rho_jacobi=0.9999, poisson_check_every=4, poisson_max_iter=20000)
    for name, w_ in (("chebyshev-sor", sor), ("multigrid-CG", wl.replace(flags=wl.flags | W.FLAG_POISSON_MG))):
        line[name] = learned_vs_plain(E, w_, args, sraw, compare_steps=max(10, args.steps // 10), trained=trained,
                                      level=L)
    print(json.dumps(line))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="pore3")
    ap.add_argument("--precision", default="f32", choices=["f32", "f64", "bf16", "fp16"])
    ap.add_argument("--cpu-budget", type=float, default=20.0)
    ap.add_argument("--replicas", type=int, default=96)
    ap.add_argument("--rho-jacobi", type=float, default=0.0,
                    help="Chebyshev spectral radius (0: library default)")
    ap.add_argument("--check-every", type=int, default=0,
                    help="Poisson residual test interval (0: workload default)")
    ap.add_argument("--poisson", default="mg", choices=["mg", "sor"],
                    help="Poisson solver: multigrid-preconditioned CG or Chebyshev red-black SOR")
    ap.add_argument("--ws-level", type=int, default=2,
                    help="lattice level of the learned warm start (--workload learned; 0: the lattice)")
    ap.add_argument("--ws-samples", type=int, default=20000,
                    help="solver snapshots the warm-start network is trained on (--workload learned)")
    ap.add_argument("--ws-iters", type=int, default=2000, help="training iterations (--workload learned)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-learned", action="store_true",
                    help="skip the learned-vs-plain warm-start comparison")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        run_reference(args)
    elif args.workload == "replicas":
        run_batch(args)
    elif args.workload == "precision":
        run_precision(args)
    elif args.workload == "learned":
        run_learned(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
