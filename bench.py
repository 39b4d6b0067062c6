"""Benchmark of the coupled D2Q9 pseudopotential + D2Q5 thermal LBM step.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Workload: the droplet-evaporation setup (open outflow, Dirichlet T = 0.95 T_c
on all edges, droplet at 0.86 T_c; Section 4.1 shape) on a 4096 x 4096
domain in FP32 -- the size the HBM-roofline target is stated on.  One step is
one coupled update of every node.  The state (2 x 1 GiB ping-pong buffers) is
larger than L2, so no flush is needed between steps.

Prints one JSON line: MLUPS (whole job), HBM roofline of the fused step
kernel (against the measured copy bandwidth, and the nominal 8 TB/s), the
end-to-end figure through the C ABI with host buffers, clocks, and the
oracle itself timed on the host cores as a baseline.  Extras (rank 0): the
FP64 step against the FP64 ALU roofline, the FP16-g variant, the 3-D form,
the D^2 law of Section 4.1 (FP32 and FP64 evaporation constants) and the
open-outflow configuration's d^2 slope, the FP32 / FP16-g field errors
against the FP64 path (which matches the oracle to 1e-10 in the tests), the
512-domain batch resident in one launch per step, and the same population
served by the continuous-batching loop.

Under torchrun (N > 1) every rank advances its own replica of the domain
(the domains are independent: replicas, weak scaling) and rank 0 reports
the aggregate over the max-over-ranks time.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import subprocess
import tempfile
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

NX = NY = 4096
BYTES_PER_NODE = {"fp32": 120, "fp64": 240, "fp32_g16": 100}
# FP64 FLOP per node update of the FP64 step (2 DFMA + DADD + DMUL thread
# instructions per node, from ncu's instruction counters on the same kernel)
# and the nominal FP64 rate of the part (no measured FP64 peak on this machine)
FP64_FLOP_PER_NODE = 239.0
FP64_NOMINAL_GFLOPS = 1250.0
METRIC = "coupled D2Q9+D2Q5 MLUPS and % of HBM roofline, FP32 vs FP64 at stated error"
STEP_SOURCES = ["paper_2205_00686_gb300/csrc/lbm_step.cu",
                "paper_2205_00686_gb300/csrc/lbm_node.cuh",
                "paper_2205_00686_gb300/csrc/lbm_internal.cuh"]
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "step_kernel_traffic.json")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=1000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true")
    ap.add_argument("--no-tune", action="store_true")
    ap.add_argument("--tile", default=None,
                    help="THREADS,ROWS: fixed tile instead of the autotuner (profiler captures)")
    ap.add_argument("--staging", default="auto", choices=["auto", "on", "off"],
                    help="load path of the FP32 step: bulk-copy staging on/off (auto: the "
                         "autotuner's choice, else on where possible)")
    ap.add_argument("--no-serve", action="store_true")
    ap.add_argument("--serve-instances", type=int, default=512)
    ap.add_argument("--serve-steps", type=int, default=5000)
    ap.add_argument("--size", type=int, default=NX,
                    help="domain side (default 4096; smaller sides for profiler captures)")
    ap.add_argument("--ny", type=int, default=None,
                    help="domain height (default: the side; profiler captures on wide, short domains)")
    ap.add_argument("--prec", default="fp32", choices=["fp32", "fp64", "fp32_g16"],
                    help="precision of the timed domain (profiler captures; the metric is FP32)")
    ap.add_argument("--zseg", type=int, default=None,
                    help="planes per CTA of the fused 3-D step (default: timed pick)")
    ap.add_argument("--only-3d", type=int, default=0, metavar="N",
                    help="run only the 3-D leg on an N^3 droplet cloud (profiler captures)")
    return ap.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def max_over_ranks(t, dist, world, device):
    """The slowest rank's time: the whole job is done when every rank is."""
    if world <= 1:
        return t
    import torch
    tt = torch.tensor([t], device=device, dtype=torch.float64)
    dist.all_reduce(tt, op=dist.ReduceOp.MAX)
    return float(tt.item())


def job_mlups(world, nodes_per_rank, steps, t):
    """Whole-job node updates per second (each rank steps its own domain)."""
    return world * nodes_per_rank * steps / t / 1e6


def step_source_hash():
    h = hashlib.sha256()
    for p in STEP_SOURCES:
        with open(os.path.join(ROOT, p), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons during a region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        # the raw samples (the JSON line carries their summary); BENCH_CLOCKS_CSV
        # names a file to keep them in
        self.path = os.environ.get("BENCH_CLOCKS_CSV") or os.path.join(
            tempfile.gettempdir(), "lbm_bench_clocks_%d.csv" % os.getpid())

    def __enter__(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + self.Q,
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=self.fh, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            time.sleep(0.2)
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self.fh.close()

    def summary(self):
        if self.proc is None or not os.path.exists(self.path):
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        sms, mx, reasons, pw = [], None, set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sms.append(float(parts[1]))
                mx = float(parts[2])
                pw.append(float(parts[3]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sms:
            return {"sm_mhz": None, "sm_max_mhz": mx, "reasons": ["no samples"]}
        return {"sm_mhz": float(np.median(sms)), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sms), "power_w_max": max(pw) if pw else None}


def make_case(n=NX, ny=None):
    from paper_2205_00686_gb300 import workloads as W
    ny = n if ny is None else ny
    return W.open_evaporation(n, ny, R=640.0 * min(n, ny) / 4096.0, steps=0)


def cpu_baseline(sample_n=1024, sample_steps=60, omp=False):
    """The FP64 C oracle on a bounded sample of the workload (a sample_n^2
    domain of the same setup): single-threaded, or (omp) its OpenMP build on
    every host core, whose results are bit-identical."""
    import oracle
    c = make_case(sample_n)
    s = oracle.Sim(c.nx, c.ny, c.params, c.bc, omp=omp)
    s.init(*c.fields())
    s.step(1)
    t0 = time.perf_counter()
    s.step(sample_steps)
    dt = time.perf_counter() - t0
    mlups = c.nx * c.ny * sample_steps / dt / 1e6
    cores = int(os.environ.get("OMP_NUM_THREADS", os.cpu_count() or 1)) if omp else 1
    return {"value": round(mlups, 3), "unit": "MLUPS", "cores": cores, "kind": "oracle",
            "sample": "%dx%d of the same setup, %d FP64 steps, %.1f s%s" % (
                c.nx, c.ny, sample_steps, dt, ", OpenMP over the per-node loops" if omp else "")}


def fritz_check(gravities=(1e-5, 2e-5, 4e-5, 8e-5), max_steps=150000):
    """Section 4.3: bubble departure from a 20-node heater at 1.1 T_c in a
    300 x 600 pool started filled with saturated liquid, FP32; the departure
    diameter per gravity (device-side region labelling every 200 steps) and
    the log-log slope (Fritz: -1/2)."""
    import paper_2205_00686_gb300 as lbm
    from paper_2205_00686_gb300 import protocols as PR
    from paper_2205_00686_gb300 import workloads as W

    def make(g):
        c = W.nucleate_boiling(300, 600, gravity=g, vapour_layer=False)
        d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec="fp32")
        d.init_fields(*c.fields())
        return d

    rg, rl = W.COEXISTENCE[0.86]
    t0 = time.perf_counter()
    out = PR.fritz_sweep(make, list(gravities), rl, rg, check_every=200, max_steps=max_steps,
                         min_area=8)
    rows = out["runs"]
    return {"setup": "Section 4.3: 300x600 pool filled with saturated liquid, 20-node heater at "
                     "1.1Tc, theta 75, lambda 2/3, open top, FP32",
            "g": list(gravities),
            "departure_step": [r["departure"]["step"] if r["departure"] else None for r in rows],
            "D_d": [round(r["departure"]["diameter"], 2) if r["departure"] else None for r in rows],
            "slope": round(out["slope"], 4) if out["slope"] is not None else None,
            "fritz_slope": -0.5, "wall_s": round(time.perf_counter() - t0, 1)}


def accuracy_check():
    """FP32 and FP32+FP16-g against FP64 on the GPU (the metric's "FP32 vs FP64
    at the stated error"): 64x64 droplet, 1000 steps, max relative field
    error.  The FP64 path's own agreement with the CPU oracle is the parity
    tests' job (<= 1e-10 on the same case)."""
    import paper_2205_00686_gb300 as lbm
    from paper_2205_00686_gb300 import workloads as W
    c = W.static_droplet()
    got = {}
    for prec in ("fp64", "fp32", "fp32_g16"):
        d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec=prec)
        d.init_fields(*c.fields())
        d.step(1000)
        got[prec] = d.get_rho_u_T()
        d.close()
    ref = got["fp64"]
    out = {p: max(float(np.abs(a - b).max() / np.abs(b).max()) for a, b in zip(got[p], ref))
           for p in ("fp32", "fp32_g16")}
    return {"case": "64x64 droplet, 1000 steps, max relative field error vs the FP64 path",
            **{k: float("%.3e" % v) for k, v in out.items()}}


def served_check(n_inst, steps, budget_gb=1.0):
    """The batched + served population: n_inst open-evaporation domains with
    sides uniform in 64..512, each advanced `steps` steps, arriving in a
    seeded Poisson stream and admitted into a 1 GB device budget; reports
    p50 / p99 time-to-N-steps and aggregate MLUPS, next to the same work run
    one domain at a time through the single-domain path."""
    import paper_2205_00686_gb300 as lbm
    from paper_2205_00686_gb300 import workloads as W
    from paper_2205_00686_gb300.serve import CudaBackend, Server
    cases = W.batch_instances(n_inst, steps=steps)
    gaps = -np.log(1.0 - W.uniform(77, n_inst)) * 0.002       # mean 2 ms between arrivals
    arrivals = [(float(t), c, steps) for t, c in zip(np.cumsum(gaps), cases)]
    be = CudaBackend("fp32", autotune_steps=3, autotune_at=32)
    srv = Server(be, mem_budget=int(budget_gb * 2 ** 30), chunk=100)
    st = srv.run(arrivals)
    nodes = sum(c.nx * c.ny for c in cases)
    # the same requests one at a time through lbm_step (first 32 of them)
    import torch
    m = min(32, n_inst)
    t0 = time.perf_counter()
    for c in cases[:m]:
        d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec="fp32")
        d.init_fields(*c.fields())
        d.step(steps)
        d.get_rho_u_T()
        d.close()
    torch.cuda.synchronize()
    t_solo = time.perf_counter() - t0
    solo_mlups = sum(c.nx * c.ny for c in cases[:m]) * steps / t_solo / 1e6
    return {"instances": n_inst, "steps_each": steps, "total_nodes": nodes,
            "budget_gb": budget_gb, "mlups": round(st["mlups"], 1),
            "mlups_at_capacity": round(st["mlups_at_capacity"], 1) if st["mlups_at_capacity"] else None,
            "p50_s": round(st["p50_s"], 4), "p99_s": round(st["p99_s"], 4),
            "wall_s": round(st["wall_s"], 2), "failed": st["failed"],
            "max_concurrent": st["max_active"],
            "sequential_single_domain_mlups": round(solo_mlups, 1)}


def d2_law_check(steps=160000, every=8000, t_fit=32000):
    """The D^2 law of Section 4.1 (200^2 box, D0 = 60 at 0.86 T_c, periodic
    flow, edges held at T_c): the evaporation constant kappa from a straight
    line fit of (D / D0)^2 against t after the initial transient, in FP32 and
    in FP64, with the fit's R^2."""
    import paper_2205_00686_gb300 as lbm
    from paper_2205_00686_gb300 import workloads as W
    out = {"setup": "Section 4.1: 200x200, D0=60 at 0.86Tc, periodic flow, T=Tc on the edges",
           "steps": steps, "fit_from_step": t_fit}
    for prec in ("fp32", "fp64"):
        c = W.d2_droplet(200, D0=60.0, T_g=1.0)
        d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec=prec)
        d.init_fields(*c.fields())
        D0 = d.diagnostics(c.rho_l, c.rho_g)["diameter"]
        t, y = [], []
        for k in range(every, steps + 1, every):
            d.step(every)
            if k >= t_fit:
                t.append(k)
                y.append((d.diagnostics(c.rho_l, c.rho_g)["diameter"] / D0) ** 2)
        d.close()
        t, y = np.array(t, float), np.array(y)
        A = np.vstack([t, np.ones_like(t)]).T
        coef = np.linalg.lstsq(A, y, rcond=None)[0]
        r2 = 1.0 - ((y - A @ coef) ** 2).sum() / ((y - y.mean()) ** 2).sum()
        out["kappa_" + prec] = float("%.5g" % -coef[0])
        out["r2_" + prec] = round(float(r2), 5)
        out["d2_ratio_end_" + prec] = round(float(y[-1]), 4)
    out["kappa_rel_diff_fp32_vs_fp64"] = float("%.3g" % abs(out["kappa_fp32"] / out["kappa_fp64"] - 1))
    return out


def d2_open_check(steps=20000, every=1000, t_fit=4000):
    """The open-outflow evaporation configuration (256^2, R = 40 at 0.86 T_c,
    edges at 0.95 T_c, zero-gradient outflow), 20 000 steps in FP32 and in
    FP64: the slope of (D / D0)^2 against t and its R^2, reported as measured
    (with these edges the droplet warms and takes in vapour rather than
    following the D^2 law, so R^2 stays well below the 0.99 of the periodic
    setup of Section 4.1)."""
    import paper_2205_00686_gb300 as lbm
    from paper_2205_00686_gb300 import workloads as W
    out = {"setup": "256x256, R=40 at 0.86Tc, edges 0.95Tc, open outflow", "steps": steps,
           "fit_from_step": t_fit}
    for prec in ("fp32", "fp64"):
        c = W.open_evaporation(256, 256)
        d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec=prec)
        d.init_fields(*c.fields())
        D0 = d.diagnostics(c.rho_l, c.rho_g)["diameter"]
        t, y = [], []
        for k in range(every, steps + 1, every):
            d.step(every)
            if k >= t_fit:
                t.append(k)
                y.append((d.diagnostics(c.rho_l, c.rho_g)["diameter"] / D0) ** 2)
        d.close()
        t, y = np.array(t, float), np.array(y)
        A = np.vstack([t, np.ones_like(t)]).T
        coef = np.linalg.lstsq(A, y, rcond=None)[0]
        r2 = 1.0 - ((y - A @ coef) ** 2).sum() / max(((y - y.mean()) ** 2).sum(), 1e-300)
        out["slope_" + prec] = float("%.5g" % coef[0])
        out["r2_" + prec] = round(float(r2), 4)
        out["d2_ratio_end_" + prec] = round(float(y[-1]), 5)
    return out


def batched_check(n_inst, steps, peak, warmup=3):
    """The batched population resident on the device: n_inst open-evaporation
    domains with sides uniform in 64..512 attached to one batch and advanced
    together, one persistent launch per step (CUDA graph replays).  Timed with
    CUDA events on the batch stream, first with the default tile, then with
    the tile lbm_batch_autotune picks on a shadow batch."""
    import torch
    import paper_2205_00686_gb300 as lbm
    from paper_2205_00686_gb300 import workloads as W
    cases = W.batch_instances(n_inst, steps=steps)
    stream = torch.cuda.Stream()
    b = lbm.Batch(stream=stream.cuda_stream)
    doms = []
    for c in cases:
        d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec="fp32", stream=stream.cuda_stream)
        d.init_fields(*c.fields())
        b.attach(d)
        doms.append(d)
    nodes = sum(c.nx * c.ny for c in cases)

    def timed(steps):
        b.step(warmup)
        b.sync()
        ev0 = torch.cuda.Event(enable_timing=True)
        ev1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        ev0.record(stream)
        b.step(steps)
        ev1.record(stream)
        ev1.synchronize()
        if b.sync() != 0:
            raise RuntimeError("batched leg: device error")
        return ev0.elapsed_time(ev1) / 1e3

    tile0 = b.tile()
    steps0 = min(steps, 500)
    t0 = timed(steps0)
    tile = b.autotune(5)
    t1 = timed(steps)
    out = {"instances": n_inst, "total_nodes": nodes, "steps": steps,
           "mlups": round(nodes * steps / t1 / 1e6, 1),
           "tile": [tile[0], tile[1]], "staged": tile[2],
           "hbm_frac_of_measured": round(BYTES_PER_NODE["fp32"] * nodes * steps / t1 / 1e9 / peak, 4),
           "default_tile": [tile0[0], tile0[1]], "default_staged": tile0[2],
           "default_tile_mlups": round(nodes * steps0 / t0 / 1e6, 1)}
    b.close()
    for d in doms:
        d.close()
    return out


def time_device(dom, steps, warmup, stream, torch, dist, world):
    dom.step(warmup)
    dom.sync()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    ev0.record(stream)
    dom.step(steps)
    ev1.record(stream)
    ev1.synchronize()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    dom.sync()
    return ev0.elapsed_time(ev1) / 1e3


def bench_3d(lbm, stream, torch, peak, n=256, steps=200, warmup=20, zseg=None):
    """The three-dimensional form (D3Q19 + D3Q7, FP32) on a 256^3 periodic
    box with a cloud of 64 droplets: GLUPS of the default (fused) step, with
    its planes per CTA picked by a short timing of a few candidates unless
    given, and the HBM fraction of the algorithmic 216 B per node update (one
    read and one write of the state); then the three-kernel step on the same
    state for comparison."""
    from paper_2205_00686_gb300 import workloads as W
    c = W.droplet_cloud3d(n, cells=max(1, n // 64))
    d = lbm.Domain3(n, n, n, c.params, c.bc, prec="fp32", stream=stream.cuda_stream)
    d.init_fields(*c.fields())
    N = n ** 3
    tried = {}
    if zseg is None:
        for zs in sorted({0, 32, 48, 64, n}):
            d.set_path(True, zs)
            tried[d.path[1]] = round(N * 10 / time_device(d, 10, 3, stream, torch, None, 1) / 1e6, 1)
        zseg = max(tried, key=tried.get)
    d.set_path(True, zseg)
    t = time_device(d, steps, warmup, stream, torch, None, 1)
    d.set_path(False)
    s3 = max(steps // 4, 10)
    t3 = time_device(d, s3, 5, stream, torch, None, 1)
    dg = d.diagnostics(c.rho_l, c.rho_g)
    d.close()
    ach = 216.0 * N / (t / steps) / 1e9
    ach3 = 216.0 * N / (t3 / s3) / 1e9
    return {"workload": "%d droplets R=16 in a %d^3 periodic box, 0.86 Tc, FP32"
                        % (max(1, n // 64) ** 3, n),
            "value": round(N * steps / t / 1e6, 1), "unit": "MLUPS", "steps": steps,
            "ms_per_step": round(t / steps * 1e3, 4), "zseg": zseg, "zseg_tried_mlups": tried,
            "roofline": {"bound": "hbm", "achieved": round(ach, 1), "peak": peak, "unit": "GB/s",
                         "frac": round(ach / peak, 4), "algorithmic_bytes_per_node": 216,
                         "kernels": "k3_macro + k3_march"},
            "three_kernels": {"mlups": round(N * s3 / t3 / 1e6, 1), "steps": s3,
                              "hbm_frac_of_measured": round(ach3 / peak, 4),
                              "kernels": "k3_macro + k3_flow + k3_thermal (+ k3_advance)"},
            "max_u_after": round(dg["max_u"], 5), "nonfinite": dg["nonfinite"]}


def run_ours(args):
    import torch
    import paper_2205_00686_gb300 as lbm
    from paper_2205_00686_gb300 import _build

    rank, world, local = dist_env()
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    # one process compiles (the objects and the library are in-tree, shared by
    # every rank); the others wait for it before loading the library
    if rank == 0:
        _build.build()
    if world > 1:
        dist.barrier()
    stream = torch.cuda.Stream()
    case = make_case(args.size, args.ny)
    N = case.nx * case.ny

    dom = lbm.Domain(case.nx, case.ny, case.params, case.bc, prec=args.prec,
                     stream=stream.cuda_stream)
    if args.tile:
        dom.set_tile(*[int(v) for v in args.tile.split(",")])
    elif not args.no_tune:
        dom.autotune(10)          # tile and load path chosen by timed trials on a scratch domain
    if args.staging != "auto":
        dom.staged = args.staging == "on"
    dom.init_fields(*case.fields())
    with ClockSampler(local) as clk:
        t = time_device(dom, args.steps, args.warmup, stream, torch, dist, world)
    t = max_over_ranks(t, dist, world, "cuda")
    mlups = job_mlups(world, N, args.steps, t)
    ms_per_step = t / args.steps * 1e3

    # end to end through the C ABI with pinned host buffers: upload the
    # fields, advance, read the fields back
    pinned = [torch.from_numpy(np.ascontiguousarray(a, np.float64)).pin_memory()
              for a in case.fields()]
    outs = [torch.empty((case.ny, case.nx), dtype=torch.float64).pin_memory() for _ in range(4)]
    e2e_steps = args.steps
    # one untimed pass of the same calls first (the first transfers to and
    # from freshly pinned buffers pay one-off mapping costs, and the step's
    # graph is captured), as the device timing has its warm-up steps
    dom.init_fields(*pinned)
    dom.step(max(args.warmup, 1))
    dom.get_rho_u_T(tuple(outs))
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    dom.init_fields(*pinned)
    dom.step(e2e_steps)
    dom.get_rho_u_T(tuple(outs))
    torch.cuda.synchronize()
    te = time.perf_counter() - t0
    te = max_over_ranks(te, dist, world, "cuda")
    e2e = {"value": round(job_mlups(world, N, e2e_steps, te), 1), "unit": "MLUPS",
           "h2d_bytes_per_step": int(4 * N * 8 / e2e_steps),
           "d2h_bytes_per_step": int(4 * N * 8 / e2e_steps),
           "call": "lbm_init_fields(host) + lbm_step(%d) + lbm_get_rho_u_T(host)" % e2e_steps,
           "untimed_passes_before": 1}

    peak, peak_kind = measured_peaks()
    algo = BYTES_PER_NODE[args.prec] * N
    achieved = algo / (t / args.steps) / 1e9   # per GPU: each rank steps its own domain
    traffic = None
    if os.path.exists(TRAFFIC_FILE):
        with open(TRAFFIC_FILE) as fh:
            tr = json.load(fh)
        if tr.get("source_hash") == step_source_hash() and tr.get("prec") == args.prec \
                and case.nx == 4096 and case.ny == 4096:
            traffic = tr.get("bytes_per_launch_4096")
    roofline = {"bound": "hbm", "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
                "frac": round(achieved / peak, 4), "traffic": traffic,
                "frac_of_nominal_8tbs": round(achieved / 8000.0, 4),
                "peak_kind": "%s hbm_gbs (copy)" % peak_kind,
                "algorithmic_bytes_per_node": BYTES_PER_NODE[args.prec],
                "kernel": "lbm::k_step<%d,%d>%s" % ({"fp64": 0, "fp32": 1, "fp32_g16": 2}[args.prec],
                                                    dom.tile()[0],
                                                    " (rows staged by bulk copies)" if dom.staged
                                                    else " (register-prefetched rows)")}

    extras = {}
    if rank == 0 and not args.no_extras:
        d64 = lbm.Domain(case.nx, case.ny, case.params, case.bc, prec="fp64",
                         stream=stream.cuda_stream)
        if not args.no_tune:
            d64.autotune(3)
        d64.init_fields(*case.fields())
        k64 = max(20, args.steps // 10)
        t64 = time_device(d64, k64, 3, stream, torch, None, 1)
        m64 = N * k64 / t64 / 1e6
        fl = FP64_FLOP_PER_NODE * m64 * 1e6 / 1e9
        extras["fp64"] = {"value": round(m64, 1), "unit": "MLUPS", "tile": list(d64.tile()),
                          "hbm_frac_of_measured": round(BYTES_PER_NODE["fp64"] * N / (t64 / k64) / 1e9 / peak, 4),
                          "roofline": {"bound": "alu", "achieved": round(fl, 1),
                                       "peak": FP64_NOMINAL_GFLOPS, "unit": "GFLOP/s",
                                       "frac": round(fl / FP64_NOMINAL_GFLOPS, 4),
                                       "peak_kind": "nominal FP64 (no measured FP64 peak)",
                                       "flop_per_node": FP64_FLOP_PER_NODE},
                          "steps": k64}
        d64.close()
        dg = lbm.Domain(case.nx, case.ny, case.params, case.bc, prec="fp32_g16",
                        stream=stream.cuda_stream)
        if not args.no_tune:
            dg.autotune(10)
        dg.init_fields(*case.fields())
        tg = time_device(dg, args.steps, 3, stream, torch, None, 1)
        extras["fp32_g16"] = {"value": round(N * args.steps / tg / 1e6, 1), "unit": "MLUPS",
                              "tile": list(dg.tile()),
                              "hbm_frac_of_measured": round(BYTES_PER_NODE["fp32_g16"] * N / (tg / args.steps) / 1e9 / peak, 4)}
        dg.close()
        extras["d3q19_d3q7"] = bench_3d(lbm, stream, torch, peak)
        extras["d2_law"] = d2_law_check()
        extras["d2_open_outflow"] = d2_open_check()
        extras["error_vs_fp64"] = accuracy_check()
        extras["fritz"] = fritz_check()
        if not args.no_serve:
            extras["batched"] = batched_check(args.serve_instances, args.serve_steps, peak)
            extras["served"] = served_check(args.serve_instances, args.serve_steps)

    cpu = cpu_omp = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline()
        cpu_omp = cpu_baseline(sample_steps=300, omp=True)

    line = {
        "metric": METRIC, "value": round(mlups, 1), "unit": "MLUPS", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms_per_step, 4),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": {"fp32": "f32", "fp64": "f64", "fp32_g16": "f32 (g stored f16)"}[args.prec],
        "data": "synthetic",
        "config": {"workload": "droplet evaporation, open outflow, Dirichlet 0.95Tc edges, "
                               "R=%g, %dx%d, %s fused step" % (640.0 * min(case.nx, case.ny) / 4096.0,
                                                               case.nx, case.ny, args.prec.upper()),
                   "nx": case.nx, "ny": case.ny,
                   "l2": "inputs larger than L2 (%.2f GiB state)"
                         % (BYTES_PER_NODE[args.prec] * N / 2 ** 30),
                   "parallelism": "replicas" if world > 1 else "single GPU",
                   "tile": list(dom.tile()), "staged": dom.staged},
        "roofline": roofline, "cpu_baseline": cpu, "cpu_baseline_all_cores": cpu_omp,
        "e2e": e2e, "clocks": clk.summary(),
        "gpu_launches": args.steps,
        **extras,
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    dom.close()
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()


def run_reference(args):
    """The FP64 CPU oracle as it stands, on the host cores, on a bounded
    sample of the same workload; rank 0 only."""
    rank, world, _ = dist_env()
    if rank != 0:
        return
    import oracle
    oracle.build()
    c = make_case(512)
    s = oracle.Sim(c.nx, c.ny, c.params, c.bc)
    s.init(*c.fields())
    for _ in range(min(args.warmup, 3)):
        s.step(1)
    steps = args.steps
    per = max(1, min(8, 200 // max(steps, 1)))   # keep the whole run to a few minutes
    t0 = time.perf_counter()
    for _ in range(steps):
        s.step(per)
    dt = time.perf_counter() - t0
    mlups = c.nx * c.ny * per * steps / dt / 1e6
    sample = "%dx%d sample of the 4096x4096 setup, %d x %d FP64 steps" % (c.nx, c.ny, steps, per)
    line = {
        "impl": "reference", "metric": METRIC, "value": round(mlups, 3), "unit": "MLUPS",
        "n_gpus": world, "steps": steps, "warmup": args.warmup,
        "ms_per_step": round(dt / steps * 1e3, 3), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "FP64 CPU oracle (single thread) on a %dx%d sample of the "
                               "droplet evaporation setup (open outflow, Dirichlet 0.95Tc edges, "
                               "R=%g)" % (c.nx, c.ny, 640.0 * c.nx / 4096.0),
                   "nx": c.nx, "ny": c.ny, "sample_of": "%dx%d" % (NX, NY)},
        "cpu_baseline": {"value": round(mlups, 3), "unit": "MLUPS", "cores": 1,
                         "kind": "oracle", "sample": sample},
        "e2e": {"value": round(mlups, 3), "unit": "MLUPS", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    if args.only_3d:
        import torch
        import paper_2205_00686_gb300 as lbm
        from paper_2205_00686_gb300 import _build
        _build.build()
        stream = torch.cuda.Stream()
        out = bench_3d(lbm, stream, torch, measured_peaks()[0], n=args.only_3d,
                       steps=args.steps, warmup=args.warmup, zseg=args.zseg)
        print(json.dumps(out), flush=True)
        return
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
