"""Benchmark of the porous (VANS) lattice Boltzmann step on GB300.

Default workload: D2Q9, 4096 x 4096 periodic domain, eps from seeded
Gaussian-smoothed noise (sigma = 16 cells) in [0.4, 1.0], tau = 0.6, Ergun
drag, body force along x, FP32 populations.  One "step" is one fused
collide-and-stream update of the whole domain (all 16.8 M cells).

Prints one JSON line: MLUPS (device time, CUDA events on the launching
stream), the roofline of the step kernel, an end-to-end figure through the
public API with host buffers, SM clocks sampled during the timed region, the
FP64 CPU oracle timed on a bounded sample, and beside the plain step the MLUPS
of the D3Q19 duct, the batched 256-domain run and the adjoint (reverse) pass.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

Under torchrun (N > 1) every rank runs the same workload on its own GPU (the
domains are independent replicas: no collective on the data path); value is
the sum over ranks, timed by the slowest rank.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "MLUPS and % of HBM-bandwidth roofline; batched and adjoint MLUPS vs plain"
WORKLOAD = ("D2Q9 4096x4096 periodic, eps smoothed noise (sigma 16) in [0.4,1.0], tau 0.6, "
            "Ergun drag (d_p 21.33) + Forchheimer, body force along x, FP32 populations")
BYTES_PER_CELL = {9: 9 * 4 * 2 + 4, 19: 19 * 4 * 2 + 4}     # algorithmic bytes per update
# operations of the D2Q9 update of kind 9 (collide_pair of vans_pair.cuh; a multiply-add
# counts two; the porosity terms, formed once per row and launch, are not counted)
FLOPS_PER_CELL = 141
# reverse step, D2Q9: lambda in and out (72), the state it reads (36), eps (4),
# the compensated eps-gradient accumulators read and written (2 x 24)
ADJ_BYTES_PER_CELL = 9 * 4 * 2 + 9 * 4 + 4 + 2 * 24
FALLBACK_HBM_GBS = 6800.0
SM_MAX_MHZ = 2070.0
REPEATS = 5       # timed regions of K steps each; value = the median region
E2E_JOBS = 6      # jobs of K steps in the end-to-end figure

# DRAM bytes per launch of the step kernel measured by ncu on the 4096^2
# workload (dram__bytes_read.sum + dram__bytes_write.sum), keyed by launch shape
# (cpt, warps, rows, kind, ctas) and a hash of the kernel sources they were
# taken on; a changed kernel or another shape reports null.
TRAFFIC = {
    # mean of two launches of an ncu capture of dram__bytes_read.sum and
    # dram__bytes_write.sum on the 4096^2 workload (one pass)
    (2, 4, 4, 9, 0, "4acf6b0186f434c5"): (705070000 + 564150000 + 705100000 + 562720000) // 2,
    (4, 4, 3, 7, 2, "beeb0982103b3064"): (677260000 + 561870000 + 677480000 + 560040000) // 2,
}
KERNEL_SOURCES = {0: "vans_step.cu", 8: "vans_cluster.cu", 9: "vans_multi.cu"}
KERNEL_SOURCES.update({k: "vans_step_tma.cu" for k in (2, 4, 5, 6, 7)})


def kernel_hash(kind: int = 2) -> str:
    """Hash of the source of this launch kind's step kernel and of the headers of this
    repository that it includes, directly or through others."""
    dirs = [os.path.join(ROOT, "paper_1406_6438_gb300", "csrc"), os.path.join(ROOT, "include")]
    h, todo, seen = hashlib.sha256(), [KERNEL_SOURCES[kind]], set()
    while todo:
        name = todo.pop(0)
        path = next(p for p in (os.path.join(d, name) for d in dirs) if os.path.exists(p))
        with open(path, "rb") as fh:
            text = fh.read()
        h.update(text)
        seen.add(name)
        for inc in re.findall(rb'^#include "(.*)"', text, re.M):
            if inc.decode() not in seen and inc.decode() not in todo:
                todo.append(inc.decode())
    return h.hexdigest()[:16]


KERNEL_NAMES = {0: "k_step<9,cpt>", 2: "k_step_tma_ring<9,32*warps,cpt>",
                4: "k_step_tma_ring<9,32*warps,cpt,warp-specialised>",
                5: "k_step_tma_ring<9,32*warps,4,contiguous,warp-specialised>",
                6: "k_step_tma_ilv<9,32*warps,cpt,strided>",
                7: "k_step_tma_ilv<9,32*warps,4,contiguous>",
                8: "k_step_cluster<9,32*warps>", 9: "k_multi<steps per launch>"}


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


def roofline(kind, cells, launch_s, steps_per_launch, sms):
    """What the step kernel reaches of what bounds it: one step per launch HBM; kind 9, whose
    launch reads and writes the state once for several steps, the FP32 pipe (rate of the
    SMs' lanes at their highest clock), with its share of HBM beside it."""
    peak, peak_kind = peaks()
    gbs = BYTES_PER_CELL[9] * cells / launch_s / 1e9
    hbm = {"achieved": gbs, "peak": peak, "unit": "GB/s", "frac": gbs / peak, "peak_kind": peak_kind}
    if kind != 9:
        return {"bound": "hbm", **hbm}
    tflops = FLOPS_PER_CELL * cells * steps_per_launch / launch_s / 1e12
    rate = sms * 128 * 2 * SM_MAX_MHZ * 1e6 / 1e12
    return {"bound": "fp32", "achieved": tflops, "peak": rate, "unit": "TFLOP/s", "frac": tflops / rate,
            "peak_kind": "SMs x 128 lanes x 2 x maximum clock", "flops_per_cell": FLOPS_PER_CELL, "hbm": hbm}


def load_balance(b, kind):
    """The load balance of one more step with per-CTA timing records: the mean over the SMs
    of their busy span / the step's makespan.  With kind 9 the profile is of the batch's
    single-step launch, not of the launches that were timed; kind 0 has none."""
    if kind == 0:
        return {}
    return {"single_step_load_balance" if kind == 9 else "load_balance": b.profile_step()}


# ------------------------------------------------------------------ clocks --
class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during a region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, dev_id: str | None):
        self.dev_id = dev_id
        self.proc = None
        self.err = None

    def __enter__(self):
        cmd = ["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits", "-lms", "100"]
        if self.dev_id:
            cmd += ["-i", self.dev_id]
        try:
            self.proc = subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.DEVNULL,
                                         text=True)
            time.sleep(0.25)
        except Exception as e:   # no nvidia-smi: report it
            self.err = str(e)
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            time.sleep(0.15)
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except Exception:
                self.proc.kill()
                out = ""
            self.lines = [ln for ln in out.splitlines() if ln.strip()]
        return False

    def summary(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "error": self.err}
        sm, smax, reasons, power = [], None, set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            c = [x.strip() for x in ln.split(",")]
            if len(c) < 9:
                continue
            try:
                sm.append(float(c[1]))
                smax = float(c[2])
                power.append(float(c[3]))
            except ValueError:
                continue
            for name, v in zip(names, c[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm),
                "power_w_max": max(power) if power else None}


def gpu_uuid(torch, dev):
    try:
        u = str(torch.cuda.get_device_properties(dev).uuid)
        return u if u.startswith("GPU-") else "GPU-" + u
    except Exception:
        return None


# ------------------------------------------------------------- CPU oracle --
def oracle_mlups(p: dict, eps: np.ndarray, budget_s: float, max_steps: int | None = None):
    """Time the FP64 oracle on (p, eps): steps until about budget_s seconds."""
    import oracle as O
    po = O.Params(**p)
    e = eps.astype(np.float64)
    f = O.init(po, e)
    t0 = time.perf_counter()
    f = O.run(po, e, f, 1)
    one = time.perf_counter() - t0
    n = max(1, int(budget_s / max(one, 1e-6)))
    if max_steps:
        n = min(n, max_steps)
    t0 = time.perf_counter()
    O.run(po, e, f, n)
    dt = time.perf_counter() - t0
    cells = p["nx"] * p["ny"] * p["nz"]
    return cells * n / dt / 1e6, n, dt, O.num_threads()


def cpu_model():
    try:
        with open("/proc/cpuinfo") as fh:
            for ln in fh:
                if ln.lower().startswith(("model name", "cpu part")):
                    return ln.split(":", 1)[1].strip()
    except Exception:
        pass
    return os.uname().machine


# -------------------------------------------------------- reference arm ----
def reference_arm(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    from paper_1406_6438_gb300 import workloads as W
    import oracle as O
    O.build()
    p, eps, _ = W.periodic_2d(4096)
    # the step of this arm: one FP64 update of a 512 x 512 periodic crop of the
    # workload's eps field (a bounded sample of the same workload)
    crop = np.ascontiguousarray(eps[:, :512, :512])
    pc = dict(p, nx=512, ny=512)
    po = O.Params(**pc)
    e = crop.astype(np.float64)
    f = O.init(po, e)
    f = O.run(po, e, f, max(args.warmup, 0))
    t0 = time.perf_counter()
    O.run(po, e, f, args.steps)
    dt = time.perf_counter() - t0
    cells = 512 * 512
    v = cells * args.steps / dt / 1e6
    line = {
        "impl": "reference", "metric": METRIC, "value": v, "unit": "MLUPS",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": dt / args.steps * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "nx": 4096, "ny": 4096,
                   "sample": "512x512 periodic crop of the 4096x4096 eps field"},
        "cpu_baseline": {"value": v, "unit": "MLUPS", "cores": O.num_threads(), "kind": "oracle",
                         "sample": f"FP64 oracle, {args.steps} steps of a 512x512 crop",
                         "cpu": cpu_model()},
        "e2e": {"value": v, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------- ranks -------
def max_over_ranks(value: float, dist, device) -> float:
    """The largest value over all ranks (each rank's timed region; the job is
    as slow as its slowest replica).  Without a process group: the value."""
    if dist is None:
        return value
    import torch
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_mlups(world: int, cells: int, steps: int, seconds: float) -> float:
    """Whole-job lattice updates per second over all replicas, in millions."""
    return world * cells * steps / seconds / 1e6


# --------------------------------------------------------------- GPU arm ---
def time_region(torch, stream, fn):
    a = torch.cuda.Event(enable_timing=True)
    b = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    a.record(stream)
    fn()
    b.record(stream)
    b.synchronize()
    return a.elapsed_time(b) / 1e3


def fixed_launch(spec):
    return None if not spec else tuple(int(v) for v in spec.split(","))


def bench_d3q19(torch, V, W, args=None):
    dims = dict(nx=256, ny=256, nz=256)
    if args is not None and args.dims:
        dims = dict(zip(("nx", "ny", "nz"), (int(v) for v in args.dims.split(","))))
    p, eps, n = W.duct_3d(**dims)
    if args is not None and args.only == "d3q19":
        n = args.steps
    s = V.Solver(p)
    s.set_eps(torch.from_numpy(eps).cuda().view(-1))
    fl = fixed_launch(args.launch) if args is not None else None
    if fl:
        s.launch = V.Launch(*fl)
        L = s.launch
    else:
        L = s.autotune()
    s.step(10)
    c0 = s.launch_count
    t = time_region(torch, s.stream, lambda: s.step(n))
    cells = p["nx"] * p["ny"] * p["nz"]
    size = "%d^3" % p["nx"] if p["nx"] == p["ny"] == p["nz"] else "%dx%dx%d" % (p["nx"], p["ny"], p["nz"])
    out = {"workload": "D3Q19 %s, walls y/z, eps noise [0.35,0.95], tau 0.6, Forchheimer" % size,
           "steps": n, "value": cells * n / t / 1e6, "unit": "MLUPS",
           "gb_s": BYTES_PER_CELL[19] * cells * n / t / 1e9,
           "launch": vars(L), "launches": s.launch_count - c0}
    out["frac_of_peak"] = out["gb_s"] / peaks()[0]
    s.close()
    return out


def bench_channel(torch, V, W, args=None):
    """The 128 x 64 porous Poiseuille channel (the parity workload): its 5000
    steps in the autotuned launch (kind 8 when one thread-block cluster holds
    the state: all of them in one launch).  The 0.6 MB state never leaves the
    chip, so the figure is MLUPS only, not an HBM fraction."""
    p, eps, n = W.channel_128x64()
    s = V.Solver(p)
    s.set_eps(torch.from_numpy(eps).cuda().view(-1))
    fl = fixed_launch(args.launch) if args is not None else None
    if fl:
        s.launch = V.Launch(*fl)
        L = s.launch
    else:
        L = s.autotune()
    if args is not None and args.only == "channel":
        n = args.steps
    s.step(64)
    c0 = s.launch_count
    t = time_region(torch, s.stream, lambda: s.step(n))
    cells = p["nx"] * p["ny"]
    out = {"workload": "D2Q9 porous Poiseuille channel 128x64, eps 0.6, Da 1e-3, tau 0.8",
           "steps": n, "value": cells * n / t / 1e6, "unit": "MLUPS", "us_per_step": t / n * 1e6,
           "launch": vars(L), "launches": s.launch_count - c0,
           "note": ("state resident on chip (kind 8: a cluster's shared memory; otherwise L2): "
                    "no HBM fraction")}
    s.close()
    return out


def bench_batched(torch, V, W, args=None):
    ndom = args.domains if args is not None and args.domains else 256
    doms = W.batched_channels(n=ndom)
    b = V.Batch([p for p, _ in doms])
    for d, (_, eps) in enumerate(doms):
        b.set_eps(d, torch.from_numpy(eps).cuda().view(-1))
    fl = fixed_launch(args.launch) if args is not None else None
    if fl:
        b.launch = V.Launch(*fl)
        L = b.launch
    else:
        L = b.autotune()
    n = args.steps if args is not None and args.only == "batched" else 2000
    b.step(20)
    c0 = b.launch_count
    t = time_region(torch, b.stream, lambda: b.step(n))
    cells = b.cells
    # a launch reads and writes the state once, whatever number of steps it takes
    per_launch = n / (b.launch_count - c0) if L.kind == 9 else 1
    out = {"workload": "256 D2Q9 channels, nx~U[64,1024], ny~U[32,512], own eps and tau",
           "domains": len(doms), "cells": cells, "steps": n,
           "value": cells * n / t / 1e6, "unit": "MLUPS",
           "gb_s": BYTES_PER_CELL[9] * cells * n / per_launch / t / 1e9,
           "launch": vars(L), "launches": b.launch_count - c0}
    out["frac_of_peak"] = out["gb_s"] / peaks()[0]
    out.update(load_balance(b, L.kind))
    b.close()
    return out


def bench_adjoint(torch, V, W, args=None):
    from paper_1406_6438_gb300.adjoint import outlet_flux
    if args is not None and args.only == "adjoint":
        p, eps, n, every = W.adjoint_channel(nsteps=args.steps, every=min(100, args.steps))
    else:
        p, eps, n, every = W.adjoint_channel()
    cells = p["nx"] * p["ny"]
    out = {"workload": "D2Q9 512x512 channel, eps noise [0.4,1.0], tau 0.8, outlet flux gradient",
           "steps": n, "checkpoint_every": every, "unit": "MLUPS (backward pass, wall clock)"}
    # FP64 central finite differences of the oracle at 32 cells of this workload
    # (a committed data file written by tests/golden/make_adjoint_fd.py)
    gold = None
    gpath = os.path.join(ROOT, "tests", "golden", "adjoint_channel_512_fd.json")
    if os.path.exists(gpath):
        with open(gpath) as fh:
            gold = json.load(fh)
        if gold.get("nsteps") != n:
            gold = None
    for bits in (32, 64):
        s = V.Solver(p)
        s.set_eps(torch.from_numpy(eps).cuda().view(-1))
        s.autotune()
        s.set_adjoint_precision(bits)
        for rep in range(2):          # the first pass allocates and captures its graphs
            e = torch.from_numpy(eps).cuda().requires_grad_(True)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            J = outlet_flux(e, s, n, every)
            torch.cuda.synchronize()
            t1 = time.perf_counter()
            c0 = s.launch_count
            J.backward()
            torch.cuda.synchronize()
            t2 = time.perf_counter()
        key = "value" if bits == 32 else "fp64_arith"
        out[key] = cells * n / (t2 - t1) / 1e6
        if bits == 32:
            out["forward_mlups"] = cells * n / (t1 - t0) / 1e6
            out["backward_launches"] = s.launch_count - c0
        out[f"grad_finite_{bits}"] = bool(torch.isfinite(e.grad).all().item())
        if gold is not None and gold["x_out"] == p["nx"] - 1:
            g = e.grad.cpu().numpy().astype(np.float64)
            fd = np.array(gold["dJdeps_fd"])
            got = np.array([g[tuple(c)] for c in gold["cells_zyx"]])
            out[f"fd_err_{bits}"] = float(np.abs(got - fd).max() / np.abs(fd).max())
        s.close()
    out["note"] = ("value: all-FP32 reverse step; fp64_arith: per-cell reverse arithmetic in FP64; "
                   "fd_err_*: max over 32 cells of |dJ/deps - FP64 FD| / max |FD|")
    if args is None or args.only != "adjoint":
        out["kernel_4096"] = bench_adjoint_kernel(torch, V, W)
    return out


def bench_adjoint_kernel(torch, V, W, n=4096, steps=40):
    """The reverse step alone on the plain step's 4096^2 workload (its buffers
    far exceed L2): K calls of vans_step_adjoint, lambda ping-ponged, timed
    with CUDA events on the solver's stream."""
    p, eps, _ = W.periodic_2d(n)
    cells = p["nx"] * p["ny"]
    s = V.Solver(p)
    s.set_eps(torch.from_numpy(eps).cuda().view(-1))
    s.step(50)
    state = s.get_state()
    lam = [s.new_state(), s.new_state()]
    grad = torch.zeros(s.grad_floats(), dtype=torch.float32, device="cuda")
    s.flux_seed(p["nx"] - 1, lam[0], grad, state)
    for k in range(3):
        s.step_adjoint(state, lam[k % 2], lam[(k + 1) % 2], grad)
    t = time_region(torch, s.stream,
                    lambda: [s.step_adjoint(state, lam[k % 2], lam[(k + 1) % 2], grad)
                             for k in range(steps)])
    out = {"workload": f"D2Q9 {n}x{n} periodic (the plain step's), reverse step alone",
           "steps": steps, "value": cells * steps / t / 1e6, "unit": "MLUPS",
           "bytes_per_cell": ADJ_BYTES_PER_CELL,
           "gb_s": ADJ_BYTES_PER_CELL * cells * steps / t / 1e9,
           "launch": "default reverse launch (kind 1: 1 cell per thread, 4 compute warps, 4 stages)",
           "finite": bool(torch.isfinite(grad).all().item())}
    out["frac_of_peak"] = out["gb_s"] / peaks()[0]
    s.close()
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="native", choices=["native", "reference"])
    ap.add_argument("--n", type=int, default=4096, help="domain edge (default 4096)")
    ap.add_argument("--no-extras", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--launch", default=None,
                    help="fixed launch shape cpt,warps,rows[,kind] instead of the autotuner")
    ap.add_argument("--only", default=None, choices=["d3q19", "batched", "adjoint", "channel"],
                    help="run one side benchmark alone (profiling captures) and print its JSON")
    ap.add_argument("--dims", default=None, help="nx,ny,nz of the D3Q19 duct for --only d3q19")
    ap.add_argument("--domains", type=int, default=0, help="domains for --only batched")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    if args.impl == "reference":
        return reference_arm(args)
    if args.only:
        import torch
        import paper_1406_6438_gb300 as V
        from paper_1406_6438_gb300 import workloads as W
        fn = {"d3q19": bench_d3q19, "batched": bench_batched, "adjoint": bench_adjoint,
              "channel": bench_channel}[args.only]
        print(json.dumps({args.only: fn(torch, V, W, args)}), flush=True)
        return 0

    import torch
    import paper_1406_6438_gb300 as V
    from paper_1406_6438_gb300 import workloads as W

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")

    p, eps, _ = W.periodic_2d(args.n)
    cells = p["nx"] * p["ny"]
    sim = V.Solver(p)
    sim.set_eps(torch.from_numpy(eps).cuda().view(-1))
    if args.launch:
        sim.launch = V.Launch(*(int(v) for v in args.launch.split(",")))
        L = sim.launch
    else:
        L = sim.autotune()
    sim.step(args.warmup)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    # REPEATS timed regions of exactly K steps each; the reported figure is
    # the median region (max over ranks), the spread is reported beside it
    regions = []
    with ClockSampler(gpu_uuid(torch, local)) as clk:
        for r in range(REPEATS):
            if dist:
                dist.barrier()
            c0 = sim.launch_count
            t_r = time_region(torch, sim.stream, lambda: sim.step(args.steps))
            launches = sim.launch_count - c0
            regions.append(max_over_ranks(t_r, dist, "cuda"))
    t = statistics.median(regions)
    ok = sim.check()
    value = job_mlups(world, cells, args.steps, t)
    sms = torch.cuda.get_device_properties(local).multi_processor_count
    roof = roofline(L.kind, cells, t / launches, args.steps / launches, sms)
    key = (L.cpt, L.warps, L.rows, L.kind, L.ctas, kernel_hash(L.kind))
    traffic = TRAFFIC.get(key) if args.n == 4096 else None

    # end to end through the public API with host buffers: E2E_JOBS jobs of K
    # steps back to back (Solver.run_jobs), each uploading its eps field from
    # pinned host memory, resetting to rest, stepping, and copying rho and u
    # back to pinned host memory; a job's copies overlap its neighbours' steps
    fields = [eps] + [W.periodic_2d(args.n, seed=100 + k)[1] for k in range(E2E_JOBS - 1)]
    eps_host = [torch.from_numpy(f).view(-1).pin_memory() for f in fields]
    rho_host = [torch.empty(cells, dtype=torch.float32).pin_memory() for _ in fields]
    u_host = [torch.empty(2 * cells, dtype=torch.float32).pin_memory() for _ in fields]
    sim.run_jobs(eps_host[:2], args.steps, rho_host[:2], u_host[:2])     # warm-up
    # REPEATS runs, the median as for the step: a run is 15 ms of host wall clock, which a
    # stall of the host doubled in 5 of 14 single ones
    e2e_runs = []
    for r in range(REPEATS):
        if dist:
            dist.barrier()
        torch.cuda.synchronize()
        w0 = time.perf_counter()
        sim.run_jobs(eps_host, args.steps, rho_host, u_host)
        e2e_runs.append(max_over_ranks(time.perf_counter() - w0, dist, "cuda"))
    t_e2e = statistics.median(e2e_runs)
    e2e_ok = bool(all(torch.isfinite(u).all().item() for u in u_host))
    h2d = cells * 4
    d2h = 3 * cells * 4
    sim.close()
    del sim
    torch.cuda.empty_cache()

    extras = {}
    cpu = None
    if world == 1 and not args.no_extras:
        for name, fn in (("channel_128x64", bench_channel), ("d3q19", bench_d3q19),
                         ("batched", bench_batched), ("adjoint", bench_adjoint)):
            try:
                extras[name] = fn(torch, V, W)
            except Exception as ex:       # report, keep the headline line
                extras[name] = {"error": repr(ex)}
            torch.cuda.empty_cache()
    if world == 1 and rank == 0 and not args.no_cpu:
        import oracle as O
        O.build()
        mlups, n_or, dt, cores = oracle_mlups(p, eps, budget_s=12.0)
        cpu = {"value": mlups, "unit": "MLUPS", "cores": cores, "kind": "oracle",
               "sample": f"FP64 oracle, {n_or} steps of the full {args.n}x{args.n} workload "
                         f"({dt:.1f} s)", "cpu": cpu_model()}
        O.set_num_threads(1)                   # the same oracle on one core
        try:
            m1, n1, dt1, _ = oracle_mlups(p, eps, budget_s=4.0, max_steps=2)
        finally:
            O.set_num_threads(cores)
        cpu["single_thread"] = {"value": m1, "unit": "MLUPS", "cores": 1,
                                "sample": f"{n1} step(s) of the same workload ({dt1:.1f} s)"}

    clocks = clk.summary()
    line = {
        "metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": t / args.steps * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic",
        "config": {"workload": WORKLOAD, "nx": args.n, "ny": args.n, "cells": cells,
                   "parallelism": "replicas" if world > 1 else "single GPU",
                   "l2": "inputs larger than L2 (two 0.6 GB population buffers), no flush",
                   "launch": vars(L)},
        "roofline": {**roof, "traffic": traffic, "bytes_per_cell": BYTES_PER_CELL[9],
                     "kernel": KERNEL_NAMES.get(L.kind, "?"), "launch_us": t / launches * 1e6,
                     "steps_per_launch": args.steps / launches},
        "e2e": {"value": job_mlups(world, cells, E2E_JOBS * args.steps, t_e2e), "unit": "MLUPS",
                "h2d_bytes_per_step": h2d / args.steps, "d2h_bytes_per_step": d2h / args.steps,
                "jobs": E2E_JOBS, "finite": e2e_ok, "runs_s": e2e_runs,
                "note": (f"median of {REPEATS} runs of {E2E_JOBS} jobs of K steps through Solver.run_jobs, host wall clock: "
                         "per job eps H2D from pinned memory, vans_set_eps_async, K steps, "
                         "vans_moments, rho+u D2H to pinned memory; copies on a second stream "
                         "overlap the neighbouring jobs' steps")},
        "gpu_launches": launches,
        "repeats": {"n": REPEATS, "ms_per_step": [r / args.steps * 1e3 for r in regions],
                    "min_ms_per_step": min(regions) / args.steps * 1e3,
                    "max_ms_per_step": max(regions) / args.steps * 1e3,
                    "note": "value is the median of the timed regions, each exactly K steps"},
        "clocks": clocks,
        "state_ok": ok,
        "cpu_baseline": cpu,
    }
    line.update(extras)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
