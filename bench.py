"""Benchmark of the solid-LBM hot path on GB300, one JSON line on stdout.

A bench step is one complete solve of the workload: reset to the rest state,
all time steps of the configuration (interior + boundary kernels each step),
then the fields (u, v, sigma) on the device.  Throughput is giga lattice
updates per second (GLUPS) over material nodes.

Default workload: the suddenly loaded edge crack on a 2048 x 2048 lattice,
crack length 512, 1500 steps, FP32 deviation storage.  Its working set
(two 151 MB distribution buffers + 67 MB displacement) exceeds the 129 MB L2,
so no L2 flush is needed between steps.  ``--workload plate`` runs the
1024 x 512 plate with a hole (20000 steps; 46 MB, L2-resident).

Arms:
  (default)          the CUDA library through its C ABI (device-resident
                     inputs), plus ``e2e`` through the same public API from
                     host buffers, ``roofline`` of the interior kernel,
                     ``cpu_baseline`` (the FP64 oracle on a bounded sample).
  --impl reference   the FP64 oracle on the host cores (bounded sample per step).

Multi-GPU (torchrun, one rank per GPU): every rank solves its own replica;
no collective on the data path ("replicas only"), weak scaling.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "GLUPS (giga lattice updates per second, whole job)"
# FP32 operations of one lattice update in the temporally blocked kernels (FMA =
# 2): moments and populations 42, 9 of them FMAs, displacement update 11
FLOPS_PER_UPDATE = 62
# with lambda != mu also the source from the density gradient (10) and its eight
# FMAs in the collision
FLOPS_PER_UPDATE_GRAD = 88
# the kernel sources each kernel's recorded DRAM traffic depends on
KERNEL_SOURCES = {"k_interior": ("lbm_kernels.cu", "lbm_device.cuh"),
                  "k_interior_pair": ("lbm_kernels.cu", "lbm_device.cuh", "lbm_pair.cuh"),
                  "k_interior_grad": ("lbm_kernels.cu", "lbm_device.cuh"),
                  "k_interior_aa": ("lbm_kernels.cu", "lbm_device.cuh"),
                  "k_tile": ("lbm_tile.cu", "lbm_async.cuh", "lbm_device.cuh"),
                  "k_tile_grad": ("lbm_tile.cu", "lbm_async.cuh", "lbm_device.cuh"),
                  "k_wave": ("lbm_wave.cu", "lbm_device.cuh"),
                  "k_wave_grad": ("lbm_wave.cu", "lbm_device.cuh")}
WORKLOADS = ("crack", "plate", "batch", "serve")


def _workload(name, material="poisson"):
    """The workload; material "paper" takes the paper's lambda != mu solid (the
    crack's c_s^2/c_d^2 = 0.3611, nu = 0.2174; the plate's c_d^2/c_s^2 = 2.8)."""
    import dataclasses
    from paper_2208_04088_gb300 import workloads as W
    if name == "crack":
        wl = W.CONFIG3
        lm = W.CRACK_PAPER_LAM_OVER_MU
    elif name == "plate":
        wl = W.CONFIG2
        lm = W.PLATE_NONPOISSON_LAM_OVER_MU
    else:
        raise SystemExit(f"unknown workload {name}")
    if material == "paper":
        wl = dataclasses.replace(wl, lam_over_mu=lm)
    return wl


def _peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.QUERY}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.thread.join(timeout=5)

    def summary(self):
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.lines:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for name, val in zip(names, parts[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax),
                "reasons": sorted(reasons), "samples": len(sm)}


def max_over_ranks(value: float, device) -> float:
    """Largest value over all ranks (the job takes as long as its slowest
    replica); identity without a process group."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    if dist.is_available() and dist.is_initialized() and dist.get_world_size() > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def _dist():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def _cpu_baseline(wl, seconds=12.0):
    """The FP64 oracle, as it stands, on the host cores: run the first steps of
    the same lattice until `seconds` have passed; GLUPS over material nodes."""
    import oracle
    nt, links = oracle.geometry(**wl.geometry_args())
    o = oracle.Oracle(nt, links, wl.bcs, lam=wl.lam, mu=wl.mu, rho0=wl.rho0, tau=wl.tau)
    nodes = int(nt.sum())
    o.step(1)  # touch memory
    steps = 0
    t0 = time.perf_counter()
    while True:
        o.step(2)
        steps += 2
        el = time.perf_counter() - t0
        if el >= seconds or steps >= wl.steps:
            break
    o.close()
    return {"value": nodes * steps / el / 1e9, "unit": "GLUPS", "cores": oracle.threads(),
            "kind": "oracle",
            "sample": f"first {steps} of {wl.steps} steps of the {wl.nx}x{wl.ny} {wl.name} "
                      f"lattice ({nodes} material nodes), {el:.1f} s"}


def run_reference(args):
    world, rank, _ = _dist()
    wl = _workload(args.workload, args.material)
    if rank != 0:
        return 0
    import oracle
    nt, links = oracle.geometry(**wl.geometry_args())
    nodes = int(nt.sum())
    per_step = max(2, int(args.ref_steps_per_step))
    o = oracle.Oracle(nt, links, wl.bcs, lam=wl.lam, mu=wl.mu, rho0=wl.rho0, tau=wl.tau)
    for _ in range(args.warmup):
        o.step(per_step)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        o.step(per_step)
    el = time.perf_counter() - t0
    o.close()
    value = nodes * per_step * args.steps / el / 1e9
    sample = (f"{per_step} time steps per bench step of the {wl.nx}x{wl.ny} {wl.name} lattice "
              f"({nodes} material nodes)")
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "GLUPS",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": el / args.steps * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": wl.name, "nx": wl.nx, "ny": wl.ny, "steps": wl.steps,
                   "storage": "f64 absolute", "l2": "host run"},
        "cpu_baseline": {"value": value, "unit": "GLUPS", "cores": oracle.threads(),
                         "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": "GLUPS", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def _sources_sha(kernel):
    """sha256 (first 16 hex) of the kernel's sources with comments and
    whitespace removed: a record stays valid across comment edits, not code
    edits."""
    import hashlib
    import re
    csrc = os.path.join(ROOT, "paper_2208_04088_gb300", "csrc")
    h = hashlib.sha256()
    for name in KERNEL_SOURCES[kernel]:
        with open(os.path.join(csrc, name)) as f:
            text = f.read()
        text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
        text = re.sub(r"//[^\n]*", " ", text)
        h.update(" ".join(text.split()).encode())
    return h.hexdigest()[:16]


def _traffic(wl, storage, kernel):
    """Measured DRAM bytes of one launch of `kernel` (profiles/traffic.json), or
    None if its sources have changed since the capture."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as f:
            t = json.load(f)[kernel]
        if t.get("sources_sha256_16") != _sources_sha(kernel):
            return None
        e = t[wl.name][storage]
        return float(e["dram_read"] + e["dram_write"])
    except (OSError, KeyError, ValueError):
        return None



def _alu_peak_tflops(dev, sm_mhz):
    """FP32 rate of the device: SMs x 128 FP32 lanes x 2 (FMA) x SM clock."""
    import torch
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    return sms * 128 * 2 * sm_mhz * 1e6 / 1e12, sms


def _blocked_kernel(time_block, lam_over_mu):
    """Name of the temporally blocked kernel: the register tiles by default (with
    lambda != mu their other form), the strips on request."""
    return ("k_wave" if time_block else "k_tile") + ("" if lam_over_mu == 1.0 else "_grad")


def _roofline_blocked(nodes, tblock, mean_launch_ms, bytes_per_update, lam_over_mu, hbm_peak,
                      hbm_kind, clk, dev):
    """Roofline of one temporally blocked launch: the HBM ceiling (one pass of
    populations and displacement per launch) and the FP32 ceiling (tblock
    updates per node); `bound` is the one with the longer minimum time."""
    fpu = FLOPS_PER_UPDATE if lam_over_mu == 1.0 else FLOPS_PER_UPDATE_GRAD
    sm_mhz = clk.get("sm_mhz") or 2070.0
    alu_peak, sms = _alu_peak_tflops(dev, sm_mhz)
    updates = nodes * tblock
    t = mean_launch_ms * 1e-3
    bytes_launch = nodes * bytes_per_update
    flops_launch = updates * fpu
    hbm = {"achieved": bytes_launch / t / 1e9, "peak": hbm_peak, "unit": "GB/s",
           "frac": bytes_launch / t / 1e9 / hbm_peak, "peak_kind": hbm_kind,
           "min_launch_us": bytes_launch / (hbm_peak * 1e9) * 1e6,
           "bytes_per_launch": bytes_launch,
           "bytes_per_update": bytes_launch / updates}
    alu = {"achieved": flops_launch / t / 1e12, "peak": alu_peak, "unit": "TFLOP/s",
           "frac": flops_launch / t / 1e12 / alu_peak,
           "peak_kind": f"derived: {sms} SMs x 128 FP32 lanes x 2 x {sm_mhz:.0f} MHz (sampled)",
           "min_launch_us": flops_launch / (alu_peak * 1e12) * 1e6,
           "flops_per_update": fpu}
    bound = "hbm" if hbm["min_launch_us"] >= alu["min_launch_us"] else "alu"
    lead = hbm if bound == "hbm" else alu
    return {"bound": bound, "achieved": lead["achieved"], "peak": lead["peak"],
            "unit": lead["unit"], "frac": lead["frac"], "peak_kind": lead["peak_kind"],
            "steps_per_launch": tblock, "updates_per_launch": updates,
            "mean_launch_ms": mean_launch_ms,
            "ceilings": {"hbm": hbm, "alu": alu},
            "bound_rule": ("the lower roofline ceiling: arithmetic intensity "
                           f"{flops_launch / bytes_launch:.2f} FLOP/B against the FP32/HBM ridge "
                           f"{alu_peak * 1e3 / hbm_peak:.2f} FLOP/B")}



def _solve_fn(solver, wl, N):
    """One bench step of a solver: reset, every time step, fields on the device."""
    import torch
    dev = solver.workspace.device
    u = torch.empty((2, wl.ny, wl.nx), device=dev)
    v = torch.empty((2, wl.ny, wl.nx), device=dev)
    sg = torch.empty((3, wl.ny, wl.nx), device=dev)

    def solve():
        solver.reset()
        solver.step(wl.steps)
        N.lbm_get_fields(solver.h, u.data_ptr(), v.data_ptr(), sg.data_ptr(), on_device=True)
    return solve


def _variant_record(wl, args, dev, stream, storage, wall_node, time_block, solves=5, warm=2):
    """Throughput of one variant of the workload (same lattice, another storage,
    wall reading or stepping form): `solves` graph-replayed solves timed with
    CUDA events on the solver's stream, then one solve in timing mode for the
    roofline of its dominant kernel."""
    import torch

    from paper_2208_04088_gb300 import _native as N
    desc = N.desc_from_workload(wl, storage=storage, wall_node=wall_node, time_block=time_block)
    nodes = int(desc.node_type.sum())
    solver = N.Solver(desc, stream=stream, device=dev)
    info = solver.info()
    solve = _solve_fn(solver, wl, N)
    for _ in range(warm):
        solve()
    solver.sync()
    torch.cuda.synchronize(dev)
    start = torch.cuda.Event(enable_timing=True)
    stop = torch.cuda.Event(enable_timing=True)
    start.record(stream)
    for _ in range(solves):
        solve()
    stop.record(stream)
    torch.cuda.synchronize(dev)
    ms = start.elapsed_time(stop)
    try:
        solver.sync()
        unstable = False
    except N.LbmError as e:
        unstable = e.status == N.LBM_ERR_UNSTABLE
        if not unstable:
            raise
    tb = int(info["time_block"])
    solver.set_timing(True)
    solver.timing()
    solver.reset()
    solver.step(wl.steps - (wl.steps % tb if tb > 1 else 0))
    tim = solver.timing()
    solver.set_timing(False)
    peak, peak_kind = _peaks()
    if tb > 1:
        mean_ms = tim["interior_ms"] / max(1, tim["steps"] // tb)
        clk = {"sm_mhz": None}  # the nominal maximum clock for this secondary record
        roof = _roofline_blocked(nodes, tb, mean_ms, info["bytes_per_update"], wl.lam_over_mu,
                                 peak, peak_kind, clk, dev)
        roof["kernel"] = _blocked_kernel(time_block, wl.lam_over_mu)
    else:
        mean_ms = tim["interior_ms"] / max(1, tim["steps"])
        gbs = info["interior_nodes"] * info["bytes_per_update"] / (mean_ms * 1e-3) / 1e9
        kname = ("k_interior_grad" if wl.lam_over_mu != 1.0 else
                 "k_interior" if storage == "f32" else "k_interior_pair")
        roof = {"bound": "hbm", "achieved": gbs, "peak": peak, "unit": "GB/s",
                "frac": gbs / peak, "peak_kind": peak_kind, "kernel": kname,
                "bytes_per_update": info["bytes_per_update"],
                "updates_per_launch": info["interior_nodes"], "mean_launch_ms": mean_ms,
                "traffic": _traffic(wl, storage, kname)}
    solver.close()
    return {"value": nodes * wl.steps * solves / (ms * 1e-3) / 1e9, "unit": "GLUPS",
            "ms_per_solve": ms / solves, "solves": solves, "storage": storage,
            "wall_values": "node" if wall_node else "extrapolate", "time_block": tb,
            "unstable": unstable, "roofline": roof}


def _batch_record(dev, stream, storage, wall_node, count, steps, loop):
    """Config 4 (seeded plates with holes, `count` instances, `steps` steps):
    one batched solve timed with CUDA events after a warm-up solve, and, if
    `loop`, the same instances solved one after another through lbm_step in
    FP32 (the per-instance loop)."""
    import torch

    from paper_2208_04088_gb300 import _native as N
    from paper_2208_04088_gb300 import workloads as W
    wls = W.batched_instances(count, seed=4, steps=steps)
    b = N.Batch([N.desc_from_workload(w, storage=storage, wall_node=wall_node) for w in wls],
                stream=stream)
    shape = b.tune(steps_per_trial=20)
    info = b.info()
    nodes = info["nodes"]
    b.reset()
    b.step(steps)
    torch.cuda.synchronize(dev)
    start = torch.cuda.Event(enable_timing=True)
    stop = torch.cuda.Event(enable_timing=True)
    start.record(stream)
    b.reset()
    b.step(steps)
    stop.record(stream)
    torch.cuda.synchronize(dev)
    ms = start.elapsed_time(stop)
    info = b.info()
    b.close()
    rec = {"value": nodes * steps / (ms * 1e-3) / 1e9, "unit": "GLUPS", "storage": storage,
           "instances": count, "material_nodes": nodes, "time_steps": steps,
           "blocked_instances": info["blocked_instances"], "unstable_instances": info["unstable"],
           "tuned_shape": shape, "ms_per_solve": ms}
    if loop:
        solvers = [N.Solver(N.desc_from_workload(w, wall_node=wall_node), stream=stream)
                   for w in wls]
        torch.cuda.synchronize(dev)
        start.record(stream)
        for sv in solvers:
            sv.step(steps)
        stop.record(stream)
        torch.cuda.synchronize(dev)
        lms = start.elapsed_time(stop)
        for sv in solvers:
            sv.close()
        rec["per_instance_loop"] = {"value": nodes * steps / (lms * 1e-3) / 1e9, "unit": "GLUPS",
                                    "storage": "f32",
                                    "how": "lbm_step per instance, one after another"}
        rec["speedup_over_loop"] = rec["value"] / rec["per_instance_loop"]["value"]
    return rec


def _k_apparent(sigma_yy, length, y):
    """Apparent stress intensity ahead of the tip (tip at x = length - 1/2):
    the largest sigma_yy sqrt(2 pi r) over r = 1.5 .. 10.5, sigma_yy averaged
    over the two rows straddling the crack plane."""
    import numpy as np
    sy = 0.5 * (np.asarray(sigma_yy[y], np.float64) + np.asarray(sigma_yy[y - 1], np.float64))
    xs = np.arange(length + 1, length + 11)
    return float((sy[xs] * np.sqrt(2 * np.pi * (xs - (length - 0.5)))).max())


def _rel_l2(a, b, mask):
    import numpy as np
    a = np.asarray(a, np.float64)[..., mask]
    b = np.asarray(b, np.float64)[..., mask]
    den = math.sqrt(float((b * b).sum()))
    return math.sqrt(float(((a - b) ** 2).sum())) / den if den > 0 else float(abs(a).max())


def _cpu_baseline_and_accuracy(wl, wall_node, dev, stream, sample_steps, t_k=500):
    """The cpu_baseline leg: the FP64 oracle, as it stands, on all host cores,
    over the whole solve of the workload.  Its first `sample_steps` steps are
    the timed sample.  Its fields at t_k and at the last step are also the
    reference of the accuracy record: the library's FP32 (default stepping
    form), FP16 and BF16 solves of the same workload against them (relative L2
    over material nodes), and the apparent stress intensity at t_k against
    Freund's K_I^0 (Sec. 5.2, valid for t < l_c/c_d)."""
    import numpy as np

    import oracle
    from paper_2208_04088_gb300 import _native as N

    gpu = {}
    for storage in ("f32", "f16", "bf16"):
        s = N.Solver(N.desc_from_workload(wl, storage=storage, wall_node=wall_node),
                     stream=stream, device=dev)
        s.step(t_k)
        a = s.fields_host()
        s.step(wl.steps - t_k)
        b = s.fields_host()
        try:
            s.sync()
        except N.LbmError:
            pass
        gpu[storage] = (a, b)
        s.close()
    nt, links = oracle.geometry(**wl.geometry_args())
    o = oracle.Oracle(nt, links, wl.bcs, lam=wl.lam, mu=wl.mu, rho0=wl.rho0, tau=wl.tau,
                      wall_node=wall_node)
    nodes = int(nt.sum())
    t0 = time.perf_counter()
    o.step(sample_steps)
    el = time.perf_counter() - t0
    cpu = {"value": nodes * sample_steps / el / 1e9, "unit": "GLUPS", "cores": oracle.threads(),
           "kind": "oracle",
           "sample": f"first {sample_steps} of {wl.steps} steps of the {wl.nx}x{wl.ny} "
                     f"{wl.name} lattice ({nodes} material nodes), {el:.1f} s; the oracle "
                     "then runs the rest of the solve for the accuracy record"}
    o.step(t_k - o.t)
    fk = o.fields()
    o.step(wl.steps - o.t)
    fl = o.fields()
    o.close()
    mask = nt.astype(bool)
    length = wl.crack[0]
    y = wl.ny // 2
    k0 = float(oracle.freund_ki0(t_k, wl.bcs[1]["value"][0], wl.nu, wl.cd))
    acc = {"reference": "FP64 oracle, same workload and wall reading",
           "t_last": wl.steps, "t_k": t_k,
           "K_I0_freund": k0, "K_apparent_oracle": _k_apparent(fk["sigma"][1], length, y)}
    for storage, (a, b) in gpu.items():
        ka = _k_apparent(a["sigma"][1], length, y)
        acc[storage] = {
            "rel_l2_t_last": {k: _rel_l2(b[k], fl[k], mask) for k in ("u", "v", "sigma")},
            "rel_l2_t_k": {k: _rel_l2(a[k], fk[k], mask) for k in ("u", "v", "sigma")},
            "K_apparent": ka,
            "K_rel_to_oracle": ka / acc["K_apparent_oracle"] - 1.0,
            "K_over_freund": ka / k0}
    return cpu, acc


def run_profile(args):
    """A short run for ncu captures: --profile N steps of the workload through
    lbm_step (replayed graphs and direct launches, as a solve) and its fields,
    then exit."""
    from paper_2208_04088_gb300 import _native as N
    import torch
    torch.cuda.set_device(0)
    wl = _workload(args.workload, args.material)
    s = N.Solver(N.desc_from_workload(wl, storage=args.storage, in_place=args.streaming == "in-place",
                                      wall_node=args.wall_values == "node",
                                      time_block=args.time_block))
    s.step(args.profile)  # as a solve does: replayed graphs, then direct launches
    s.fields_host()
    s.close()
    print(json.dumps({"profile_steps": args.profile, "workload": wl.name,
                      "storage": args.storage}), flush=True)
    return 0


def run_batch(args):
    """Config 4: 256 seeded plate-with-hole instances, 5000 steps each, advanced
    together by the batched persistent launch (autotuned shape, replayed
    graphs); beside it the same instances solved one after another through
    lbm_step in FP32 (the per-instance loop)."""
    import torch

    from paper_2208_04088_gb300 import _native as N
    from paper_2208_04088_gb300 import workloads as W

    world, rank, local = _dist()
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    N.load(build_if_missing=False)
    wls = W.batched_instances(args.batch_count, seed=4, steps=args.batch_steps)
    stream = torch.cuda.Stream(device=dev)
    wall_node = args.wall_values == "node"
    descs = [N.desc_from_workload(w, storage=args.storage, wall_node=wall_node,
                                  in_place=args.streaming == "in-place") for w in wls]
    b = N.Batch(descs, stream=stream)
    shape = b.tune(steps_per_trial=20)
    nodes = b.info()["nodes"]

    def barrier():
        torch.cuda.synchronize(dev)
        if world > 1:
            torch.distributed.barrier()

    for _ in range(args.warmup):
        b.reset()
        b.step(args.batch_steps)
    barrier()
    start = torch.cuda.Event(enable_timing=True)
    stop = torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clocks:
        barrier()
        start.record(stream)
        for _ in range(args.steps):
            b.reset()
            b.step(args.batch_steps)
        stop.record(stream)
        barrier()
    unstable = b.info()["unstable"]
    blocked = b.info()["blocked_instances"]
    ms = start.elapsed_time(stop)
    ms = max_over_ranks(ms, dev)
    value = nodes * args.batch_steps * args.steps * world / (ms * 1e-3) / 1e9
    launches = b.info()["kernel_launches"]
    b.close()

    # the per-instance FP32 loop over the same instances (one pass)
    loop = None
    if not args.no_loop:
        s_loop = torch.cuda.Event(enable_timing=True)
        e_loop = torch.cuda.Event(enable_timing=True)
        solvers = [N.Solver(N.desc_from_workload(w, wall_node=wall_node), stream=stream)
                   for w in wls]
        barrier()
        s_loop.record(stream)
        for sv in solvers:
            sv.step(args.batch_steps)
        e_loop.record(stream)
        barrier()
        lms = s_loop.elapsed_time(e_loop)
        loop = {"value": nodes * args.batch_steps / (lms * 1e-3) / 1e9, "unit": "GLUPS",
                "storage": "f32", "how": "lbm_step per instance, one after another"}
        for sv in solvers:
            sv.close()
    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "GLUPS", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": ms / args.steps,
            "bench_step": (f"one batched solve: reset, {args.batch_steps} time steps of every "
                           "instance"),
            "ms_per_time_step": ms / args.steps / args.batch_steps,
            "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": args.storage, "data": "synthetic",
            "config": {"workload": f"batched_{len(wls)}_hole_plates_seed4",
                       "instances": len(wls), "material_nodes": nodes,
                       "time_steps": args.batch_steps, "storage": args.storage + " deviations",
                       "wall_values": args.wall_values, "tuned_shape": shape,
                       "parallelism": f"replicas x{world}",
                       "l2": "inputs larger than L2"},
            "unstable_instances": unstable,
            "blocked_instances": blocked,
            "per_instance_loop": loop,
            "clocks": clocks.summary(), "gpu_launches": int(launches),
            "roofline": None, "e2e": None, "cpu_baseline": None,
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


def _serve_trace(trace, storage, wall_node, budget_gb, tick_steps, in_place=False, gpu=0):
    """Serve a seeded request trace (arrival time, workload) with the
    continuous-batching server: requests are submitted when their arrival time
    has passed on the wall clock, ticks run while any request is live.  Latency
    runs from arrival to fields on the host; aggregate GLUPS is the work of all
    requests over the makespan."""
    import torch

    from paper_2208_04088_gb300 import _native as N
    from paper_2208_04088_gb300 import workloads as W

    stream = torch.cuda.Stream()
    srv = N.Server(int(budget_gb * (1 << 30)), storage=storage, stream=stream)
    # warm the kernels and the graph on a small request
    wid = srv.submit(N.desc_from_workload(W.square_plate(64, 0), storage=storage,
                                          wall_node=wall_node), 64)
    while srv.result(wid) is None:
        srv.tick(tick_steps)
    lat = []
    lu = 0
    unstable = 0
    pending = list(trace)
    live = {}
    t0 = time.perf_counter()
    with ClockSampler(gpu) as clocks:
        while pending or live:
            now = time.perf_counter() - t0
            while pending and pending[0][0] <= now:
                at, w = pending.pop(0)
                d = N.desc_from_workload(w, storage=storage, wall_node=wall_node,
                                         in_place=in_place)
                live[srv.submit(d, w.steps)] = (at, w.nodes * w.steps)
            if not live:
                time.sleep(min(0.01, max(0.0, pending[0][0] - now)))
                continue
            srv.tick(tick_steps)
            for rid in list(live):
                r = srv.result(rid)
                if r is not None:
                    unstable += int(r["unstable"])
                    at, work = live.pop(rid)
                    lat.append(time.perf_counter() - t0 - at)
                    lu += work
    makespan = time.perf_counter() - t0
    srv.close()
    lat = sorted(lat)
    p50 = lat[len(lat) // 2]
    p99 = lat[min(len(lat) - 1, int(math.ceil(0.99 * len(lat))) - 1)]
    return {"value": lu / makespan / 1e9, "unit": "GLUPS", "requests": len(lat),
            "latency_s": {"p50": p50, "p99": p99, "max": lat[-1]},
            "unstable_requests": unstable, "makespan_s": makespan,
            "storage": storage, "clocks": clocks.summary()}


def run_serve(args):
    """Config 5: a seeded trace of solve requests with Poisson arrivals, served
    by the continuous-batching server under an HBM budget; p50/p99 latency from
    arrival to fields-on-host, and aggregate GLUPS over the makespan."""
    import torch

    from paper_2208_04088_gb300 import _native as N
    from paper_2208_04088_gb300 import workloads as W

    torch.cuda.set_device(0)
    N.load(build_if_missing=False)
    trace = W.serving_trace(args.requests, seed=5, rate=args.rate,
                            max_side=args.max_side, max_steps=args.max_steps)
    r = _serve_trace(trace, args.storage, args.wall_values == "node", args.budget_gb,
                     args.tick_steps, in_place=args.streaming == "in-place")
    line = {
        "metric": METRIC, "value": r["value"], "unit": "GLUPS", "n_gpus": 1,
        "steps": r["requests"], "warmup": 1,
        "ms_per_step": r["makespan_s"] / r["requests"] * 1e3,
        "bench_step": "one served request (makespan / requests)",
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": args.storage, "data": "synthetic",
        "config": {"workload": f"serving_trace_seed5_rate{args.rate:g}_n{r['requests']}",
                   "rate_per_s": args.rate, "requests": r["requests"],
                   "sides": f"64..{args.max_side} (powers of two)",
                   "steps": f"1000..{args.max_steps} log-uniform",
                   "budget_gb": args.budget_gb, "tick_steps": args.tick_steps,
                   "storage": args.storage + " deviations", "wall_values": args.wall_values},
        "latency_s": r["latency_s"],
        "unstable_requests": r["unstable_requests"],
        "makespan_s": r["makespan_s"], "clocks": r["clocks"],
        "roofline": None, "e2e": None, "cpu_baseline": None,
    }
    print(json.dumps(line), flush=True)
    return 0


def run_gpu(args):
    import numpy as np
    import torch

    from paper_2208_04088_gb300 import _native as N

    world, rank, local = _dist()
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    N.load(build_if_missing=False)
    wl = _workload(args.workload, args.material)
    stream = torch.cuda.Stream(device=dev)

    wall_node = args.wall_values == "node"
    desc = N.desc_from_workload(wl, storage=args.storage, wall_node=wall_node,
                                time_block=args.time_block, in_place=args.streaming == "in-place")
    nodes = int(desc.node_type.sum())
    solver = N.Solver(desc, stream=stream, device=dev)
    info0 = solver.info()
    fields = {"u": torch.empty((2, wl.ny, wl.nx), device=dev),
              "v": torch.empty((2, wl.ny, wl.nx), device=dev),
              "s": torch.empty((3, wl.ny, wl.nx), device=dev)}

    def solve():
        solver.reset()
        solver.step(wl.steps)
        N.lbm_get_fields(solver.h, fields["u"].data_ptr(), fields["v"].data_ptr(),
                         fields["s"].data_ptr(), on_device=True)

    def barrier():
        torch.cuda.synchronize(dev)
        if world > 1:
            torch.distributed.barrier()

    for _ in range(args.warmup):
        solve()
    solver.sync()
    barrier()

    # timed region 1 (the value): the production path, replayed CUDA graphs with
    # the boundary kernel on a side branch
    launches0 = solver.info()["kernel_launches"]
    start = torch.cuda.Event(enable_timing=True)
    stop = torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clocks:
        barrier()
        start.record(stream)
        for _ in range(args.steps):
            solve()
        stop.record(stream)
        barrier()
    solver.sync()
    elapsed_ms = start.elapsed_time(stop)
    launches = solver.info()["kernel_launches"] - launches0
    elapsed_ms = max_over_ranks(elapsed_ms, dev)
    total_lu = nodes * wl.steps * args.steps * world
    value = total_lu / (elapsed_ms * 1e-3) / 1e9

    # timed region 2 (the kernel durations): with every launch bracketed by
    # CUDA events on its own stream (library timing mode: direct launches).
    # One step per launch: the whole solves, interior and boundary kernels.
    # Temporally blocked: the solves' blocked launches (a multiple of the block).
    tblock = int(info0["time_block"])
    n_timed = max(1, min(args.steps, args.timing_solves))
    solver.set_timing(True)
    solver.timing()  # clear
    barrier()
    start.record(stream)
    for _ in range(n_timed):
        if tblock > 1:
            solver.reset()
            solver.step(wl.steps - wl.steps % tblock)
        else:
            solve()
    stop.record(stream)
    barrier()
    tim = solver.timing()
    timing_ms = start.elapsed_time(stop)
    solver.set_timing(False)
    peak, peak_kind = _peaks()
    clk = clocks.summary()
    if tblock > 1:
        # temporally blocked kernel: one launch carries tblock steps of every
        # node with one HBM pass.  Two roofline ceilings bound its launch time:
        # HBM (the algorithmic bytes of one pass, bytes_per_update per node,
        # against the measured copy peak) and FP32 arithmetic (the algorithmic
        # operations of tblock updates per node, FMA = 2, against SMs x 128
        # lanes x 2 x the sampled SM clock).  The bound is the ceiling that
        # allows the smaller throughput, i.e. the longer minimum launch time.
        n_launch = max(1, tim["steps"] // tblock)
        mean_launch_ms = tim["interior_ms"] / n_launch
        kname = _blocked_kernel(args.time_block, wl.lam_over_mu)
        roofline = _roofline_blocked(nodes, tblock, mean_launch_ms, info0["bytes_per_update"],
                                     wl.lam_over_mu, peak, peak_kind, clk, dev)
        roofline.update({
            "traffic": args.traffic if args.traffic is not None else _traffic(wl, args.storage, kname),
            "kernel": kname,
            "timing": (f"events around every blocked launch over {n_timed} solves "
                       f"({tim['steps']} steps) in timing mode; that pass ran at "
                       f"{timing_ms / max(1, tim['steps']) * 1e3:.1f} us/step vs "
                       f"{elapsed_ms / args.steps / wl.steps * 1e3:.1f} us/step "
                       "for the graph-replayed value")})
    else:
        # one step per launch: the interior kernel is HBM-bound; algorithmic
        # bytes per launch / mean launch time
        bpu = info0["bytes_per_update"]
        interior = info0["interior_nodes"]
        mean_interior_ms = tim["interior_ms"] / max(1, tim["steps"])
        achieved_gbs = interior * bpu / (mean_interior_ms * 1e-3) / 1e9
        kname = ("k_interior_grad" if wl.lam_over_mu != 1.0 else
                 "k_interior_aa" if args.streaming == "in-place" else
                 "k_interior" if args.storage == "f32" else "k_interior_pair")
        roofline = {"bound": "hbm", "achieved": achieved_gbs, "peak": peak,
                    "unit": "GB/s", "frac": achieved_gbs / peak,
                    "traffic": args.traffic if args.traffic is not None else _traffic(wl, args.storage, kname),
                    "kernel": kname,
                    "bytes_per_update": bpu, "updates_per_launch": interior,
                    "mean_launch_ms": mean_interior_ms, "peak_kind": peak_kind,
                    "boundary_kernel_ms_per_step": tim["boundary_ms"] / max(1, tim["steps"]),
                    "timing": (f"events around every launch over {n_timed} solves "
                               f"({tim['steps']} steps) in timing mode; that pass ran at "
                               f"{timing_ms / n_timed / wl.steps * 1e3:.1f} us/step vs "
                               f"{elapsed_ms / args.steps / wl.steps * 1e3:.1f} us/step "
                               "for the graph-replayed value")}

    # end to end through the public API from host buffers: create (host tables
    # -> device), all steps, fields -> pinned host buffers, destroy
    e2e = None
    if not args.no_e2e:
        from concurrent.futures import ThreadPoolExecutor
        host_u = torch.empty((2, wl.ny, wl.nx), pin_memory=True)
        host_v = torch.empty((2, wl.ny, wl.nx), pin_memory=True)
        host_s = torch.empty((3, wl.ny, wl.nx), pin_memory=True)
        h2d = None
        e2e_streams = [torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)]

        def e2e_create(k):
            # host tables -> a solver on its own stream: geometry, classification,
            # device allocation, table uploads
            nonlocal h2d
            d = N.desc_from_workload(wl, storage=args.storage, wall_node=wall_node,
                                     time_block=args.time_block,
                                     in_place=args.streaming == "in-place")
            h = N.lbm_create(d, e2e_streams[k % 2].cuda_stream, 0, 0)
            inf = N.lbm_get_info(h)
            h2d = (inf["pitch"] * wl.ny + 16 * inf["boundary_nodes"] +
                   128 * inf["boundary_nodes"] + 24 * len(wl.bcs))
            return h

        def e2e_finish(h):
            N.lbm_step(h, wl.steps)
            N.lbm_get_fields(h, host_u.data_ptr(), host_v.data_ptr(), host_s.data_ptr(),
                             on_device=False)
            N.lbm_destroy(h)

        e2e_finish(e2e_create(0))  # warm-up: kernels loaded, launch plan cached
        barrier()
        n_e2e = max(1, min(args.steps, 5))
        # solves back to back as a service would run them: the host prepares
        # solve k + 1 (on a worker thread, its own stream) while the GPU steps
        # solve k; every solve's create, uploads, steps, field download and
        # destroy lie inside the timed region
        with ThreadPoolExecutor(1) as pool:
            t0 = time.perf_counter()
            fut = pool.submit(e2e_create, 0)
            for k in range(n_e2e):
                h = fut.result()
                if k + 1 < n_e2e:
                    fut = pool.submit(e2e_create, k + 1)
                e2e_finish(h)
            barrier()
            el = time.perf_counter() - t0
        el = max_over_ranks(el, dev)
        e2e = {"value": nodes * wl.steps * n_e2e * world / el / 1e9, "unit": "GLUPS",
               "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(7 * 4 * wl.nx * wl.ny),
               "steps": n_e2e,
               "includes": "lbm_create from host tables (classification, device allocation, "
                           "H2D), lbm_step, lbm_get_fields to pinned host, lbm_destroy; "
                           "solve k + 1 created on a host thread while solve k steps"}

    solver.close()

    # the rest of the metric, measured in the same run (rank 0, one GPU only):
    # the other wall reading, FP16 storage, a served trace, and the FP64
    # oracle's run of the same solve (the cpu_baseline leg) with the accuracy
    # of the FP32, FP16 and BF16 solves against it
    extras = {}
    cpu = None
    if rank == 0 and world == 1 and not args.no_extras and args.workload == "crack":
        extras["paper_rule"] = _variant_record(wl, args, dev, stream, args.storage,
                                               wall_node=not wall_node,
                                               time_block=args.time_block)
        extras["fp16"] = _variant_record(wl, args, dev, stream, "f16", wall_node=wall_node,
                                         time_block=1)
        from paper_2208_04088_gb300 import workloads as W
        trace = W.serving_trace(args.sub_requests, seed=5, rate=args.sub_rate,
                                max_side=args.sub_max_side, max_steps=args.sub_max_steps)
        extras["batch"] = {
            "workload": f"batched_{args.batch_count}_hole_plates_seed4, {args.batch_steps} steps",
            "f32": _batch_record(dev, stream, "f32", wall_node, args.batch_count,
                                 args.batch_steps, loop=True),
            "f16": _batch_record(dev, stream, "f16", wall_node, args.batch_count,
                                 args.batch_steps, loop=False)}
        extras["serving"] = {
            "trace": (f"seed 5, {args.sub_requests} requests, Poisson {args.sub_rate:g}/s, "
                      f"sides 64..{args.sub_max_side}, steps 1000..{args.sub_max_steps}; "
                      "150 GB budget, 256 steps per tick"),
            "f32": _serve_trace(trace, "f32", wall_node, 150.0, 256, gpu=local),
            "f16": _serve_trace(trace, "f16", wall_node, 150.0, 256, gpu=local)}
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        if args.no_extras or args.workload != "crack":
            cpu = _cpu_baseline(wl, seconds=args.cpu_seconds)
        else:
            cpu, extras["accuracy"] = _cpu_baseline_and_accuracy(
                wl, wall_node, dev, stream, sample_steps=args.cpu_sample_steps)
    if rank == 0:
        esz = 4 if args.storage == "f32" else 2
        nbuf = 1 if args.streaming == "in-place" else 2  # population buffers
        line = {
            "metric": METRIC, "value": value, "unit": "GLUPS", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": elapsed_ms / args.steps,
            "bench_step": (f"one solve: reset, {wl.steps} time steps of the whole lattice, "
                           "fields on the device"),
            "ms_per_time_step": elapsed_ms / args.steps / wl.steps,
            "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": args.storage,
            "data": "synthetic",
            "config": {"workload": wl.name, "nx": wl.nx, "ny": wl.ny, "time_steps": wl.steps,
                       "lambda_over_mu": wl.lam_over_mu,
                       "material_nodes": nodes, "storage": args.storage + " deviations",
                       "wall_values": args.wall_values, "streaming": args.streaming,
                       "parallelism": f"replicas x{world}",
                       "l2": ("inputs larger than L2 (working set "
                              f"{(nbuf * 9 * esz + 16) * wl.nx * wl.ny / 1e6:.0f} MB)"
                              if (nbuf * 9 * esz + 16) * wl.nx * wl.ny > 129e6 else
                              "working set fits in L2; no flush inside a solve")},
            "roofline": roofline,
            "time_block": tblock,
            "clocks": clk,
            "gpu_launches": int(launches),
            "e2e": e2e,
            "cpu_baseline": cpu,
        }
        line.update(extras)
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--workload", default="crack", choices=WORKLOADS)
    ap.add_argument("--storage", default="f32", choices=["f32", "f16", "bf16"])
    ap.add_argument("--material", default="poisson", choices=["poisson", "paper"],
                    help="poisson: lambda = mu (nu = 1/4); paper: the paper's lambda != mu "
                         "solid of the workload (crack nu = 0.2174, plate c_d^2/c_s^2 = 2.8)")
    ap.add_argument("--wall-values", default="node", choices=["extrapolate", "node"],
                    help="Neumann wall values: the boundary node's own (default) or the "
                         "paper's extrapolation along the link, whose density mode grows "
                         "after ~700 steps of the crack and dominates the fields by 1500")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=12.0,
                    help="oracle sample length when the accuracy record is not taken")
    ap.add_argument("--cpu-sample-steps", type=int, default=500,
                    help="timed oracle steps of the cpu_baseline leg (it then runs the rest "
                         "of the solve untimed for the accuracy record)")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the paper-rule, FP16, serving and accuracy records")
    ap.add_argument("--sub-requests", type=int, default=40)
    ap.add_argument("--sub-rate", type=float, default=10.0)
    ap.add_argument("--sub-max-side", type=int, default=1024)
    ap.add_argument("--sub-max-steps", type=int, default=20000)
    ap.add_argument("--timing-solves", type=int, default=3,
                    help="solves of the second timed pass that times each kernel launch")
    ap.add_argument("--ref-steps-per-step", type=int, default=4)
    ap.add_argument("--batch-count", type=int, default=256)
    ap.add_argument("--batch-steps", type=int, default=5000)
    ap.add_argument("--no-loop", action="store_true", help="batch: skip the per-instance loop")
    ap.add_argument("--rate", type=float, default=2.0, help="serve: mean arrivals per second")
    ap.add_argument("--requests", type=int, default=60)
    ap.add_argument("--max-side", type=int, default=2048)
    ap.add_argument("--max-steps", type=int, default=50000)
    ap.add_argument("--budget-gb", type=float, default=150.0)
    ap.add_argument("--tick-steps", type=int, default=256)
    ap.add_argument("--time-block", type=int, default=0,
                    help="steps per launch: 0 library default, 1 one-step kernels, "
                         "8 temporally blocked kernel")
    ap.add_argument("--streaming", choices=("two-buffers", "in-place"), default="two-buffers",
                    help="population streaming: two buffers, or one buffer in place (AA pattern, "
                         "one step per launch)")
    ap.add_argument("--profile", type=int, default=0,
                    help="run this many direct-launch steps of the workload and exit (for ncu)")
    ap.add_argument("--traffic", type=float, default=None,
                    help="ncu dram bytes per interior launch, if measured for this kernel")
    args = ap.parse_args()
    if args.impl == "reference":
        return run_reference(args)
    if args.profile:
        return run_profile(args)
    if args.workload == "batch":
        return run_batch(args)
    if args.workload == "serve":
        return run_serve(args)
    return run_gpu(args)


if __name__ == "__main__":
    sys.exit(main())
