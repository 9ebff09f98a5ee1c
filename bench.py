#!/usr/bin/env python
"""Benchmark: finite-T OF-DFT molecular dynamics on GB300.

Workload (default): 128 H at 1.0 g/cm^3, 31.25 kK, 96^3 grid, ftGGA (VT84F) +
PZ LDA, FP64, velocity Verlet (0.2 fs) with a Nose-Hoover thermostat and
density extrapolation; one step = one MD step (ion update, v_ext and Ewald,
CG minimisation to ||dF/dphi|| < 1e-8, forces, pressure).  Metric: MD steps/s.

  python bench.py --gpus N --steps K --warmup W [--impl reference]

N > 1 runs independent replicas (one per rank, launched by torchrun); value
is the steps of all ranks over the slowest rank's time (weak scaling).
--impl reference times the FP64 CPU oracle on bounded samples of the same
workload and prints the same metric.
"""
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

# Energy + potential evaluations per step of the FP64 CG (the same
# algorithm, decision for decision, in the oracle and on the GPU), as the GPU
# arm of this script measures them on each workload (its evals_per_step:
# 632-636 per MD step of md-vt84f-96 in its recent runs, 334 for md-sga-96,
# 550 per solve of solve-vt84f-128).  The reference arm runs without the
# GPU path, so it converts the oracle's measured evaluations/s with these;
# mixed workloads use the FP64 count, since the oracle is FP64 throughout.
EVALS_PER_STEP = {"md-vt84f-96": 634.0, "md-sga-96": 334.0, "md-vt84f-96-mixed": 634.0,
                  "solve-vt84f-128": 550.0, "solve-vt84f-128-mixed": 550.0, "eval-vt84f-128": 1.0}

# Arithmetic of each precision form.  FP64 contexts keep every field in
# binary64 in HBM and compute FFTs, G-space terms and the pointwise
# functional in double-float (two binary32 words, about 48 significant
# bits) on the FP32 units; reductions, CG scalars, Ewald, forces and the
# integrator run in binary64.  Mixed contexts run the field kernels in
# binary32 (per-thread partial sums in double-float, binary64 above) and
# finish in an FP64 context's arithmetic.
DTYPE = {"fp64": "f64 (double-float compute, binary64 storage and reductions)",
         "mixed": "f32 fields + f64 (f32 FFTs/pointwise, f64 reductions, double-float FP64 polish)",
         "binary64": "f64 (binary64 evaluation)"}

WORKLOADS = {
    "md-vt84f-96": dict(kind="md", functional="vt84f", grid=96, precision="fp64"),
    "md-sga-96": dict(kind="md", functional="sga", grid=96, precision="fp64"),
    "md-vt84f-96-mixed": dict(kind="md", functional="vt84f", grid=96, precision="mixed"),
    # one energy + potential evaluation per step (256 H, 4 g/cm^3, 128^3, 250 kK)
    "eval-vt84f-128": dict(kind="eval", functional="vt84f", grid=128, precision="fp64"),
    # one single-point minimisation per step (256 H, 4 g/cm^3, 128^3, 250 kK)
    "solve-vt84f-128": dict(kind="solve", functional="vt84f", grid=128, precision="fp64", T=2.5e5),
    "solve-vt84f-128-mixed": dict(kind="solve", functional="vt84f", grid=128, precision="mixed", T=2.5e5),
    # the same solve by truncated Newton (central-difference Hessian products)
    "solve-vt84f-128-tn": dict(kind="solve", functional="vt84f", grid=128, precision="fp64", T=2.5e5,
                               method="tn"),
    # batched form: 64 uneven single-point solves (8-512 H, 0.1-10 g/cm^3,
    # 2 kK-4 MK, 32^3-160^3, ftTF/SGA/VT84F) per step, all in flight at once
    "batch-64-mixed": dict(kind="batch", precision="mixed", count=64),
    "batch-64-fp64": dict(kind="batch", precision="fp64", count=64),
    # serving form: Poisson arrivals (50/s) of EOS requests, each an initial
    # minimisation and 5 VT84F MD steps (16-128 H, 0.1-20 g/cm^3, <= 96^3)
    "serve-eos-mixed": dict(kind="serve", precision="mixed", count=24, md_steps=5),
    # the same stream at the large end of the serving range: 6 requests of
    # 128-1024 H at 0.03-2 g/cm^3, grids 96^3-256^3 (not part of the default
    # line: minutes of device time with its sequential FP64 comparison)
    "serve-eos-large-mixed": dict(kind="serve", precision="mixed", count=6, md_steps=5, seed=7,
                                  n_range=(128, 1024), rho_range=(0.03, 2.0), grid_hi=256),
}


def workload_meta(name):
    """Metric, unit and config of a workload (shared by both arms)."""
    from paper_1406_0835_gb300 import inputs
    wl = WORKLOADS[name]
    if wl["kind"] == "md":
        cfg = inputs.config_md(wl["functional"], grid=wl["grid"])
        conf = {"workload": name, "atoms": len(cfg["Z"]), "grid": list(cfg["grid"]),
                "functional": wl["functional"], "xc": "PZ81", "T_K": cfg["T"], "rho_gcc": 1.0,
                "dt_fs": 0.2, "gtol": 1e-8, "l2": "flushed (256 MB write) before every timed step"}
        return "MD steps/s", "MD steps/s", conf
    if wl["kind"] == "solve":
        cfg = inputs.config_mixed(wl["T"], grid=wl["grid"])
        conf = {"workload": name, "atoms": len(cfg["Z"]), "grid": list(cfg["grid"]),
                "functional": wl["functional"], "xc": "PZ81", "T_K": cfg["T"], "rho_gcc": 4.0,
                "gtol": 1e-8, "start": "uniform density",
                "l2": "flushed (256 MB write) before every timed step"}
        return "single-point solves/s", "solves/s", conf
    cfg = inputs.config_mixed(2.5e5, grid=wl["grid"])
    conf = {"workload": name, "atoms": len(cfg["Z"]), "grid": list(cfg["grid"]),
            "functional": wl["functional"], "T_K": cfg["T"], "rho_gcc": 4.0,
            "l2": "flushed (256 MB write) before every timed step"}
    return "functional+grad evals/s", "evals/s", conf


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="md-vt84f-96", choices=sorted(WORKLOADS))
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-ref", action="store_true",
                    help="batch/serve workloads: skip the sequential FP64 reference run")
    ap.add_argument("--no-extra", action="store_true",
                    help="MD workloads: skip the sub-records (binary64 and mixed-precision MD, "
                         "batched form, serving form) that the default line carries")
    ap.add_argument("--maxit", type=int, default=20000,
                    help="CG iteration cap per solve (solve workloads; a small cap makes a short "
                         "profiling case, whose solves then stop unconverged)")
    return ap.parse_args()


def read_peaks():
    """The machine's measured peaks; the profiling recipe's fallback (6.8 TB/s,
    1.9 PFLOP/s bf16) when the file is absent."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            d = json.load(f)
            d["source"] = "measured"
            return d
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "source": "fallback"}


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device=0):
        self.device = device
        self.rows = []
        self.proc = None
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.device), "--query-gpu=" + self.FIELDS,
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 9:
                self.rows.append(parts)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        if self.thread:
            self.thread.join(timeout=2)
        sm = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in self.rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in self.rows for k in range(4)
                          if r[5 + k].lower() in ("active", "1")})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(self.rows)}


def fft_flops(n):
    return 5.0 * n * math.log2(n)


# Pointwise FP64 work per grid point of the GGA functional + PZ81 (table
# polynomials of xi, zeta, A, B and their t-derivatives, two enhancement
# factors with their s^2-derivatives, n^(-1/3), PZ81, W and the energy
# densities): about 150-250 flop per point; 200 is used.
POINTWISE_FLOP = 200.0
# Issued warp instructions and DRAM bytes per grid point of one k_pw<DD>
# launch (the FP64 contexts' pointwise kernel, VT84F at an MD density, 96^3),
# from the ncu capture summarised in profiles/k_pw_dd_96.md (67,088,952
# warp instructions, 29.96 MB per launch).  Valid for that kernel only: set
# to None when it changes until the capture is repeated.
PW_DD_WARP_INST_PER_POINT = 67088952.0 / 96 ** 3
PW_DD_TRAFFIC_PER_POINT = (28.412032e6 + 1.549440e6) / 96 ** 3
# FP32-unit instructions per FP64-equivalent flop of the double-float
# arithmetic in the cost model of the FFT and pointwise work: a sum
# (two_sum + tail + fast_two_sum) takes 11, a product (two_prod + two FMAs
# + fast_two_sum) 9, about two sums per product: 10.3.
DD_INSTR_PER_FLOP = (2 * 11 + 9) / 3.0


def kernel_model(name, g, fttf=False, real_basis=False):
    """Algorithmic FLOPs and HBM bytes of one timed launch (FP64 fields) of a
    kernel class: transforms as FFTs, 5 n log2 n per complex line (two real
    lines travel as one complex line), plus the pointwise functional; bytes =
    fields read + written once.  real_basis: the classes of the tensor-core
    form (edges up to 144), where a class of two launches of different kinds
    counts their mean."""
    nx, ny, nz = g
    K = nz // 2 + 1
    N = nx * ny * nz
    NH = nx * ny * K

    def real(n):               # one transform of a real field along an axis of n points
        return N / (2.0 * n) * fft_flops(n)

    if name == "pw":           # pointwise functional: phi, 3 derivatives in; v_part, 3 U out
        flops = POINTWISE_FLOP * N
        byts = 8 * N * 8
    elif real_basis and name == "dline":   # n -> 3 derivatives and z coefficients; 3 U -> their derivatives
        three = 2 * (real(nx) + real(ny) + real(nz))
        flops = real(nz) if fttf else three + real(nz) / 2
        byts = 8 * N * (2 if fttf else 5.5)
    elif real_basis and name == "ypass":   # y forward or inverse: coefficients in and out
        flops = real(ny)
        byts = 8 * N * 2
    elif real_basis and name == "xhl":     # x forward, Hartree and local terms, x inverse
        flops = 2 * real(nx)
        byts = 8 * N * 3
    elif real_basis and name == "zfwd":    # density: phi in, n out
        flops = N
        byts = 8 * N * 2
    elif real_basis and name == "zfinal":  # z inverse; GGA also v from v_HL, v_part, 3 derivatives, phi
        flops = real(nz) if fttf else real(nz) / 2
        byts = 8 * N * (2 if fttf else 4.5)
    elif name == "dline":      # one derivative along x or y: forward + inverse line transforms
        flops = real(nx) + real(ny)
        byts = 8 * N * 2                                   # field in, derivative out
    elif name == "zfinal":     # GGA: U_z forward + one inverse; ftTF: inverse + pointwise
        # GGA fields: U_z, v_part, d_y U_y, d_x U_x, phi in; v out
        flops = real(nz) * (1 if fttf else 2) + (POINTWISE_FLOP * N if fttf else 0)
        byts = 16 * NH + 8 * N * (3 if fttf else 6)
    elif name == "ypass":
        flops = nx * K * fft_flops(ny)
        byts = 16 * NH * 2
    elif name == "xhl":
        flops = 2 * ny * K * fft_flops(nx)
        byts = 16 * NH * 3
    else:
        flops, byts = 0.0, 0.0
    return flops, byts


def run_eval(args, rank, world):
    """Functional + gradient evaluations/s: one energy + potential
    evaluation per step at a fixed random density (inputs resident)."""
    import numpy as np
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1406_0835_gb300 import inputs, ofdft
    wl = WORKLOADS[args.workload]
    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    stream = torch.cuda.Stream(device=dev)
    cfg = inputs.config_mixed(2.5e5, grid=wl["grid"])
    ctx = ofdft.Context(cfg["L"], cfg["grid"], cfg["ions"], cfg["Z"], cfg["T"], wl["functional"],
                        precision=wl["precision"], device=dev, stream=stream.cuda_stream)
    ctx.autotune(reps=8)
    # a partly minimised density (60 CG iterations from the uniform start)
    # is the realistic input; the evaluation repeats at it
    ctx.minimize(gtol=1e-8, maxit=60, raise_on_noconv=False)
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")
    for _ in range(args.warmup):
        ofdft.ofdft_energy_potential(ctx.ctx, None, False)
    torch.cuda.synchronize()
    times = []
    with torch.cuda.stream(stream):
        for _ in range(args.steps):
            flush.fill_(1.0)
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            ofdft.ofdft_energy_potential(ctx.ctx, None, False)
            e1.record(stream)
            e1.synchronize()
            times.append(e0.elapsed_time(e1) / 1e3)
    t = sum(times)
    res = {"metric": "functional+grad evals/s", "value": world * args.steps / t,
           "unit": "evals/s", "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
           "ms_per_step": 1e3 * t / args.steps, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": DTYPE[wl["precision"]], "data": "synthetic",
           "config": {"workload": args.workload, "atoms": len(cfg["Z"]), "grid": list(cfg["grid"]),
                      "functional": wl["functional"], "T_K": cfg["T"], "rho_gcc": 4.0,
                      "l2": "flushed (256 MB write) before every timed step"}}
    ctx.close()
    return res, 1.0


def roofline_entry(dominant, grid, kms, kcount, clk, peaks, precision="fp64"):
    """Roofline position of the dominant kernel class.  On FP64 contexts the
    pointwise kernel runs double-float arithmetic on the FP32 units and is
    bound by instruction issue: achieved = its issued instructions (warp
    instructions per grid point from the ncu capture x 32 lanes x points)
    over the mean CUDA-event-timed launch; peak = 152 SMs x 4 schedulers x
    32 lanes x the median SM clock of the timed region.  The model figures
    beside it: FP64-equivalent TFLOP/s of the algorithmic flops (FFT flops +
    200 flop per point for the pointwise functional) against the issue rate
    over DD_INSTR_PER_FLOP, and against the FP64 units' peak."""
    flops, byts = kernel_model(dominant, grid, real_basis=precision == "fp64" and max(grid) <= 144)
    avg_s = (kms / 1e3) / max(kcount, 1)
    sm_mhz = clk.get("sm_mhz") or peaks.get("sm_max_mhz", 2070.0)
    issue = 152 * 128 * (sm_mhz * 1e6)                      # thread instructions / s
    dd_peak = issue / DD_INSTR_PER_FLOP / 1e12              # FP64-equivalent TFLOP/s (model)
    fp64_peak = 152 * 2 * 2 * (sm_mhz * 1e6) / 1e12         # the FP64 units: 2 DFMA / SM / clock
    ok = kcount > 0
    npts = grid[0] * grid[1] * grid[2]
    flops_rate = flops / avg_s / 1e12 if ok else None
    measured = dominant == "pw" and precision == "fp64" and PW_DD_WARP_INST_PER_POINT is not None
    out = {"bound": "alu", "kernel": dominant, "launches": kcount, "avg_launch_us": avg_s * 1e6,
           "algorithmic_flops": flops, "algorithmic_bytes": byts,
           "hbm_gbs": byts / avg_s / 1e9 if ok else None, "hbm_peak_gbs": peaks.get("hbm_gbs"),
           "hbm_peak_source": peaks.get("source"),
           "fp64_equiv_tflops": flops_rate, "fp64_equiv_model_peak": dd_peak,
           "frac_model": flops_rate / dd_peak if ok else None, "fp64_unit_peak": fp64_peak,
           "timed_launches": "FP64 and FP32 launches of the class averaged" if precision == "mixed" else "FP64"}
    if measured and ok:
        inst = PW_DD_WARP_INST_PER_POINT * 32 * npts
        out.update({"achieved": inst / avg_s / 1e12, "peak": issue / 1e12,
                    "unit": "T thread-instructions/s (issue, FP32 units)",
                    "frac": inst / avg_s / issue, "traffic": PW_DD_TRAFFIC_PER_POINT * npts,
                    "instructions_per_launch": inst,
                    "peak_note": "peak = 152 SMs x 128 lanes x median SM clock; instructions per launch "
                                 "from ncu (smsp__inst_executed x 32), time from CUDA events"})
    else:
        out.update({"achieved": flops_rate, "peak": dd_peak,
                    "unit": "TFLOP/s (FP64-equivalent, double-float on the FP32 units)",
                    "frac": out["frac_model"], "traffic": None,
                    "peak_note": "peak = 152 SMs x 128 lanes x median SM clock / %.1f FP32 instructions "
                                 "per FP64-equivalent flop" % DD_INSTR_PER_FLOP})
    return out


def time_dominant(ctx, ofdft, dominant, stream, work):
    """Average duration of the dominant kernel class: events on the launching
    stream around each of its launches during one more (host-driven) step."""
    import torch
    ofdft.ofdft_timer_select(ctx.ctx, dominant)
    ofdft.ofdft_timer_read(ctx.ctx, reset=True)
    with torch.cuda.stream(stream):
        work()
    torch.cuda.synchronize()
    kms, kcount = ofdft.ofdft_timer_read(ctx.ctx, reset=True)
    ofdft.ofdft_timer_select(ctx.ctx, 0)
    return kms, kcount


def max_over_ranks(x, world):
    """Largest x over the ranks (the slowest rank's time).  Replicas exchange
    only this scalar, on the process group's device (GPU for NCCL, host for
    gloo)."""
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    tt = torch.tensor([x], device=dev, dtype=torch.float64)
    dist.all_reduce(tt, op=dist.ReduceOp.MAX)
    return float(tt.item())


def replica_throughput(units_per_rank, seconds, world):
    """Whole-job throughput of independent replicas (weak scaling): the units
    every rank processed over the slowest rank's time.  Returns (value, time)."""
    t = max_over_ranks(seconds, world)
    return world * units_per_rank / t, t


def run_ours(args, rank, world):
    """MD workloads: one step = one MD step (ions, v_ext, Ewald, CG
    minimisation, forces, pressure, thermostat)."""
    import numpy as np
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1406_0835_gb300 import inputs, ofdft

    wl = WORKLOADS[args.workload]
    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    stream = torch.cuda.Stream(device=dev)
    cfg = inputs.config_md(wl["functional"], grid=wl["grid"])
    mdT = cfg["T"]

    def prepared_context():
        c = ofdft.Context(cfg["L"], cfg["grid"], cfg["ions"], cfg["Z"], cfg["T"], wl["functional"],
                          precision=wl["precision"], device=dev, stream=stream.cuda_stream)
        c.autotune(reps=8)       # launch shapes for this grid (cached per process)
        # step 0: minimise at the initial geometry and compute forces
        c.md_step(0.2, mdT, nsteps=0, pos=cfg["ions"], vel=cfg["vel"])
        for _ in range(args.warmup):
            c.md_step(0.2, mdT, nsteps=1)
        return c

    ctx = prepared_context()
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")   # 256 MB > L2
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    dominant = "pw" if wl["functional"] != "fttf" else "zfinal"
    launches0 = ctx.kernel_launches()
    clocks = ClockSampler(dev)
    clocks.start()
    times = []
    evals = iters = 0
    with torch.cuda.stream(stream):
        for _ in range(args.steps):
            flush.fill_(1.0)                              # evict L2 between timed steps
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            out = ctx.md_step(0.2, mdT, nsteps=1)
            e1.record(stream)
            e1.synchronize()
            times.append(e0.elapsed_time(e1) / 1e3)
            evals += out["stats"]["evaluations"]
            iters += out["stats"]["iterations"]
    torch.cuda.synchronize()
    clk = clocks.stop()
    launches = ctx.kernel_launches() - launches0
    value, t_total = replica_throughput(args.steps, sum(times), world)
    kms, kcount = time_dominant(ctx, ofdft, dominant, stream, lambda: ctx.md_step(0.2, mdT, nsteps=1))
    ctx.close()
    # End to end through the C ABI with host position and velocity buffers
    # every step: a second context replays the same trajectory (the path is
    # deterministic), so the timed steps do the same CG work as above.
    e2e = None
    if not args.no_e2e:
        ctx2 = prepared_context()
        pos, vel = ctx2.md_state()
        t_e2e = 0.0
        evals2 = 0
        for _ in range(args.steps):
            flush.fill_(1.0)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            out = ctx2.md_step(0.2, mdT, nsteps=1, pos=pos, vel=vel)
            t_e2e += time.perf_counter() - t0
            pos, vel = out["pos"], out["vel"]
            evals2 += out["stats"]["evaluations"]
        ctx2.close()
        nat = len(cfg["Z"])
        e2e = {"value": world * args.steps / max_over_ranks(t_e2e, world), "unit": "MD steps/s",
               "h2d_bytes_per_step": 2 * nat * 3 * 8,
               "d2h_bytes_per_step": 3 * nat * 3 * 8 + 16 * 8,
               "evals_per_step": evals2 / args.steps}
    res = {"metric": "MD steps/s", "value": value, "unit": "MD steps/s", "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * t_total / args.steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": DTYPE[wl["precision"]],
           "data": "synthetic (seeded hydrogen, random positions and Maxwell-Boltzmann velocities)",
           "config": {"workload": args.workload, "atoms": len(cfg["Z"]), "grid": list(cfg["grid"]),
                      "functional": wl["functional"], "xc": "PZ81", "T_K": mdT, "rho_gcc": 1.0,
                      "dt_fs": 0.2, "gtol": 1e-8, "parallelism": "replicas" if world > 1 else "single GPU",
                      "l2": "flushed (256 MB write) before every timed step",
                      "launch_shapes": "ofdft_autotune before step 0"},
           "evals_per_s": world * evals / t_total, "evals_per_step": evals / args.steps,
           "cg_iterations_per_step": iters / args.steps,
           "gpu_launches": launches, "clocks": clk, "e2e": e2e,
           "roofline": roofline_entry(dominant, cfg["grid"], kms, kcount, clk, read_peaks(), wl["precision"])}
    if world == 1 and not args.no_extra:
        res["extra"] = extra_records(args, cfg, wl, dev, stream)
    return res, evals / args.steps


def md_rate(cfg, wl, dev, stream, steps, warmup, precision, pointwise="f32x2", gtol=1e-8):
    """MD steps/s of another arithmetic (or per-step tolerance) on the same
    workload: a fresh context, step 0 and `warmup` steps untimed, then
    `steps` steps timed with CUDA events on the context's stream (L2 flushed
    before each)."""
    import torch
    from paper_1406_0835_gb300 import ofdft
    c = ofdft.Context(cfg["L"], cfg["grid"], cfg["ions"], cfg["Z"], cfg["T"], wl["functional"],
                      precision=precision, pointwise=pointwise, device=dev, stream=stream.cuda_stream)
    c.autotune(reps=8)
    c.md_step(0.2, cfg["T"], nsteps=0, pos=cfg["ions"], vel=cfg["vel"], gtol=gtol)
    for _ in range(warmup):
        c.md_step(0.2, cfg["T"], nsteps=1, gtol=gtol)
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    t, evals, evals_lo = 0.0, 0, 0
    with torch.cuda.stream(stream):
        for _ in range(steps):
            flush.fill_(1.0)
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            out = c.md_step(0.2, cfg["T"], nsteps=1, gtol=gtol)
            e1.record(stream)
            e1.synchronize()
            t += e0.elapsed_time(e1) / 1e3
            evals += out["stats"]["evaluations"]
            evals_lo += out["stats"]["evaluations_lo"]
    E = out["E"]
    c.close()
    return {"value": steps / t, "unit": "MD steps/s", "steps": steps, "warmup": warmup,
            "ms_per_step": 1e3 * t / steps, "evals_per_step": evals / steps,
            "fp32_evals_per_step": evals_lo / steps, "dtype": DTYPE[precision if pointwise != "f64" else "binary64"],
            "gtol": gtol, "F_tot_last": E["F_tot"]}


def extra_records(args, cfg, wl, dev, stream):
    """Sub-records of the default line: the same MD workload in binary64
    and in mixed precision, the batched form and the serving form, each with
    its plain-FP64 comparator, so that one run carries every part of the
    metric (MD steps/s, evals/s, batched solves/s, served p50/p99)."""
    import copy
    out = {}
    out["binary64_md"] = md_rate(cfg, wl, dev, stream, steps=3, warmup=1, precision="fp64", pointwise="f64")
    if wl["precision"] == "fp64":
        out["mixed_md"] = md_rate(cfg, wl, dev, stream, steps=5, warmup=2, precision="mixed")
        # the mixed form at the serving form's per-step tolerance (its
        # stated bars against FP64: tests/test_gpu_md_forms.py)
        from paper_1406_0835_gb300 import ofdft
        out["mixed_md_serving_gtol"] = md_rate(cfg, wl, dev, stream, steps=5, warmup=2, precision="mixed",
                                               gtol=ofdft.MIXED_MD_GTOL)
    for name, fn in (("batch-64-mixed", run_batch), ("serve-eos-mixed", run_serve)):
        a = copy.copy(args)
        a.workload, a.steps, a.warmup, a.no_ref = name, 2, 1, False
        r, _ = fn(a, 0, 1)
        keep = ("metric", "value", "unit", "steps", "warmup", "ms_per_step", "dtype", "config", "converged",
                "completed", "evals_per_step", "fp32_evals_per_step", "p50_latency_s", "p99_latency_s",
                "peak_running", "reference_fp64", "clocks", "gpu_launches")
        out[name] = {k: r[k] for k in keep if k in r}
    return out


def run_solve(args, rank, world):
    """Single-point workloads: one step = one free-energy minimisation from
    the uniform start to ||g|| < 1e-8, then forces and pressure (256 H at
    4 g/cm^3, 250 kK, 128^3, VT84F + PZ81)."""
    import numpy as np
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1406_0835_gb300 import inputs, ofdft

    wl = WORKLOADS[args.workload]
    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    stream = torch.cuda.Stream(device=dev)
    cfg = inputs.config_mixed(wl["T"], grid=wl["grid"])
    ctx = ofdft.Context(cfg["L"], cfg["grid"], cfg["ions"], cfg["Z"], cfg["T"], wl["functional"],
                        precision=wl["precision"], device=dev, stream=stream.cuda_stream)
    ctx.autotune(reps=8)

    def solve(c):
        c.set_phi(None)
        if wl.get("method") == "tn":
            E, st, nh = c.minimize_tn(gtol=1e-8, maxit=min(args.maxit, 500), raise_on_noconv=args.maxit >= 20000)
            st["hessian_products"] = nh
        else:
            E, st = c.minimize(gtol=1e-8, maxit=args.maxit, raise_on_noconv=args.maxit >= 20000)
        F, P = c.forces()
        return st

    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")
    for _ in range(args.warmup):
        solve(ctx)
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    launches0 = ctx.kernel_launches()
    clocks = ClockSampler(dev)
    clocks.start()
    times, evals, evals_lo, iters = [], 0, 0, 0
    with torch.cuda.stream(stream):
        for _ in range(args.steps):
            flush.fill_(1.0)
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            st = solve(ctx)
            e1.record(stream)
            e1.synchronize()
            times.append(e0.elapsed_time(e1) / 1e3)
            evals += st["evaluations"]
            evals_lo += st["evaluations_lo"]
            iters += st["iterations"]
    torch.cuda.synchronize()
    clk = clocks.stop()
    launches = ctx.kernel_launches() - launches0
    t_total = max_over_ranks(sum(times), world)
    dominant = "pw" if wl["functional"] != "fttf" else "zfinal"
    kms, kcount = time_dominant(ctx, ofdft, dominant, stream, lambda: solve(ctx))
    e2e = None
    if not args.no_e2e:
        # public API with host buffers: ion positions in, forces and pressure out
        t_e2e = 0.0
        for _ in range(args.steps):
            flush.fill_(1.0)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ctx.set_positions(cfg["ions"])
            solve(ctx)
            t_e2e += time.perf_counter() - t0
        nat = len(cfg["Z"])
        e2e = {"value": world * args.steps / max_over_ranks(t_e2e, world), "unit": "solves/s",
               "h2d_bytes_per_step": nat * 3 * 8, "d2h_bytes_per_step": nat * 3 * 8 + 8 + 16 * 8}
    ctx.close()
    res = {"metric": "single-point solves/s", "value": world * args.steps / t_total, "unit": "solves/s",
           "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
           "ms_per_step": 1e3 * t_total / args.steps, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": DTYPE[wl["precision"]],
           "data": "synthetic (seeded hydrogen, random positions)",
           "config": {"workload": args.workload, "atoms": len(cfg["Z"]), "grid": list(cfg["grid"]),
                      "functional": wl["functional"], "xc": "PZ81", "T_K": cfg["T"], "rho_gcc": 4.0,
                      "gtol": 1e-8, "start": "uniform density",
                      "parallelism": "replicas" if world > 1 else "single GPU",
                      "l2": "flushed (256 MB write) before every timed step"},
           "evals_per_step": evals / args.steps, "fp32_evals_per_step": evals_lo / args.steps,
           "iterations_per_step": iters / args.steps, "method": wl.get("method", "cg"),
           "evals_per_s": world * evals / t_total,
           "gpu_launches": launches, "clocks": clk, "e2e": e2e,
           "roofline": roofline_entry(dominant, cfg["grid"], kms, kcount, clk, read_peaks(), wl["precision"])}
    return res, evals / args.steps


def run_batch(args, rank, world):
    """Batched form: one step = the 64 single-point solves of the uneven batch
    (each from the uniform start to ||g|| < 1e-8), started together on 64
    streams (one graph launch each) and waited for together.  The same
    instances solved one after another with FP64 contexts are timed once as
    the plain-FP64 reference."""
    import numpy as np
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1406_0835_gb300 import inputs, ofdft

    wl = WORKLOADS[args.workload]
    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    systems = inputs.config_batch(count=wl["count"])
    ctxs = [ofdft.Context(d["L"], d["grid"], d["ions"], d["Z"], d["T"], d["functional"],
                          precision=wl["precision"], device=dev) for d in systems]
    t0 = time.perf_counter()
    for c in ctxs:
        c.autotune(reps=2)
    t_tune = time.perf_counter() - t0

    gtol = ofdft.MIXED_FORM_GTOL if wl["precision"] == "mixed" else 1e-8

    def batch_step():
        for c in ctxs:
            c.set_phi(None)
        E, S, st = ofdft.ofdft_batch_minimize([c.ctx for c in ctxs], gtol=gtol, maxit=20000)
        return E, S, st

    for _ in range(args.warmup):
        batch_step()
    torch.cuda.synchronize()
    launches0 = sum(c.kernel_launches() for c in ctxs)
    clocks = ClockSampler(dev)
    clocks.start()
    times = []
    evals = evals_lo = 0
    for _ in range(args.steps):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        E, S, st = batch_step()
        torch.cuda.synchronize()
        times.append(time.perf_counter() - t0)
        evals += sum(x["evaluations"] for x in S)
        evals_lo += sum(x["evaluations_lo"] for x in S)
    clk = clocks.stop()
    launches = sum(c.kernel_launches() for c in ctxs) - launches0
    nconv = sum(1 for x in S if x["status"] == 0)
    FP = [c.forces() for c in ctxs]            # accuracy check, outside the timed region
    for c in ctxs:
        c.close()
    t_total = sum(times)
    value = wl["count"] * args.steps / t_total
    ref = None
    if not args.no_ref:
        # plain FP64 path, one instance after another
        t_ref = t_same = 0.0
        dF, dFor, dP = [], [], []
        for d, e, (Fm, Pm) in zip(systems, E, FP):
            with ofdft.Context(d["L"], d["grid"], d["ions"], d["Z"], d["T"], d["functional"],
                               precision="fp64", device=dev) as c:
                c.minimize(gtol=1e-8, maxit=1, raise_on_noconv=False)          # graph build
                if gtol != 1e-8:
                    # context: plain FP64 to the batch's own (looser) tolerance
                    c.set_phi(None)
                    torch.cuda.synchronize()
                    t0 = time.perf_counter()
                    c.minimize(gtol=gtol, maxit=20000, raise_on_noconv=False)
                    torch.cuda.synchronize()
                    t_same += time.perf_counter() - t0
                c.set_phi(None)
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                Er, Sr = c.minimize(gtol=1e-8, maxit=20000, raise_on_noconv=False)
                torch.cuda.synchronize()
                t_ref += time.perf_counter() - t0
                Fr, Pr = c.forces()
                dF.append(abs(Er["F_tot"] - e["F_tot"]) / len(d["Z"]))
                dFor.append(float(np.max(np.abs(Fr - Fm))))
                dP.append(abs(Pr - Pm) / max(abs(Pr), 1e-30))
        ref = {"fp64_sequential_solves_per_s": wl["count"] / t_ref, "fp64_gtol": 1e-8,
               "speedup": value * t_ref / wl["count"], "max_abs_dF_per_atom_Ha": max(dF),
               "max_abs_dforce_Ha_bohr": max(dFor), "max_rel_dP": max(dP)}
        if t_same > 0.0:
            ref["fp64_sequential_same_gtol_solves_per_s"] = wl["count"] / t_same
            ref["speedup_same_gtol"] = value * t_same / wl["count"]
    grids = sorted({d["grid"][0] for d in systems})
    res = {"metric": "batched solves/s", "value": value, "unit": "solves/s", "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * t_total / args.steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": DTYPE[wl["precision"]],
           "data": "synthetic (seeded hydrogen instances)",
           "config": {"workload": args.workload, "instances": wl["count"], "grid_edges": grids,
                      "atoms": [min(len(d["Z"]) for d in systems), max(len(d["Z"]) for d in systems)],
                      "functionals": sorted({d["functional"] for d in systems}), "gtol": gtol,
                      "l2": "inputs (all instances) larger than L2"},
           "converged": nconv, "evals_per_step": evals / args.steps,
           "fp32_evals_per_step": evals_lo / args.steps, "autotune_s": t_tune,
           "gpu_launches": launches, "clocks": clk, "reference_fp64": ref}
    return res, evals / args.steps


def run_serve(args, rank, world):
    """Serving form: EOS requests arrive as a Poisson stream (50/s); each is an
    initial minimisation plus md_steps VT84F MD steps on its own context; the
    server admits them by HBM footprint into up to 8 slots.  Reports p50/p99
    latency (submit to result) and throughput, and the same requests run one
    at a time on FP64 contexts."""
    import numpy as np
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1406_0835_gb300 import inputs, ofdft

    wl = WORKLOADS[args.workload]
    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    n_range, grid_hi = wl.get("n_range", (16, 128)), wl.get("grid_hi", 96)
    rho_range = wl.get("rho_range", (0.1, 20.0))
    stream = inputs.config_serve(count=wl["count"], seed=wl.get("seed", 6), n_range=n_range,
                                 rho_range=rho_range, grid_hi=grid_hi)

    def serve(precision, slots, paced):
        with ofdft.Server(max_slots=slots, device=dev) as s:
            ids = []
            start = s.clock()
            for t_arr, d in stream:
                if paced:
                    while s.clock() - start < t_arr:
                        time.sleep(0.0005)
                ids.append(s.submit(d["L"], d["grid"], d["ions"], d["Z"], d["T"], "vt84f", precision,
                                    md_steps=wl["md_steps"], dt_fs=0.2, vel=d["vel"], maxit=20000,
                                    gtol=ofdft.MIXED_MD_GTOL if precision == "mixed" else 1e-8))
            s.drain()
            res = [s.poll(i) for i in ids]
            peak = s.peaks()
        lat = np.array([r["t_done"] - r["t_submit"] for r in res])
        span = max(r["t_done"] for r in res) - min(r["t_submit"] for r in res)
        return res, lat, span, peak

    # warm-up: one small request per precision (library load, first graphs)
    with ofdft.Server(max_slots=1, device=dev) as s:
        d = stream[0][1]
        for p in (wl["precision"], "fp64"):
            s.submit(d["L"], d["grid"], d["ions"], d["Z"], d["T"], "vt84f", p, md_steps=1, vel=d["vel"])
        s.drain()
    clocks = ClockSampler(dev)
    clocks.start()
    res, lat, span, peak = serve(wl["precision"], 8, True)
    clk = clocks.stop()
    ok = sum(1 for r in res if r["status"] == 0)
    ref = None
    if not args.no_ref:
        rres, rlat, rspan, _ = serve("fp64", 1, False)
        dF = max(abs(a["E"]["F_tot"] - b["E"]["F_tot"]) / len(d["Z"])
                 for a, b, (_, d) in zip(res, rres, stream))
        ref = {"fp64_sequential_requests_per_s": len(stream) / rspan,
               "fp64_sequential_p50_s": float(np.percentile(rlat, 50)),
               "fp64_sequential_p99_s": float(np.percentile(rlat, 99)),
               "speedup": (len(stream) / span) / (len(stream) / rspan),
               "max_abs_dF_per_atom_Ha": dF}
    value = len(stream) / span
    out = {"metric": "served requests/s", "value": value, "unit": "requests/s", "n_gpus": world,
           "steps": len(stream), "warmup": 1, "ms_per_step": 1e3 * span / len(stream),
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": DTYPE[wl["precision"]],
           "data": "synthetic (seeded Poisson EOS request stream)",
           "config": {"workload": args.workload, "requests": len(stream), "rate_per_s": 50.0,
                      "md_steps": wl["md_steps"], "slots": 8, "grid_max": grid_hi,
                      "grids": sorted({d["grid"][0] for _, d in stream}),
                      "gtol": ofdft.MIXED_MD_GTOL, "fp64_gtol": 1e-8,
                      "atoms": list(n_range), "rho_gcc": list(rho_range), "T_K": [2e3, 4e6]},
           "p50_latency_s": float(np.percentile(lat, 50)), "p99_latency_s": float(np.percentile(lat, 99)),
           "completed": ok, "peak_admitted_bytes": peak[0], "peak_running": peak[1],
           "evaluations": int(sum(r["evaluations"] for r in res)),
           "clocks": clk, "reference_fp64": ref}
    return out, 1.0


def oracle_system(args):
    """The oracle's System for the workload, and its metric unit."""
    import oracle as O
    from paper_1406_0835_gb300 import inputs
    wl = WORKLOADS[args.workload]
    if wl["kind"] == "solve":
        cfg, unit = inputs.config_mixed(wl["T"], grid=wl["grid"]), "solves/s"
    elif wl["kind"] == "eval":
        cfg, unit = inputs.config_mixed(2.5e5, grid=wl["grid"]), "evals/s"
    else:
        cfg, unit = inputs.config_md(wl["functional"], grid=wl["grid"]), "MD steps/s"
    so = O.System(cfg["L"], cfg["grid"], cfg["ions"], cfg["Z"], cfg["T"], wl["functional"])
    return so, cfg, unit


def oracle_sample(args, so, phi, evals_per_step, budget_s):
    """One bounded sample of the oracle's own CG minimiser on the full-size
    workload: CG iterations (each one energy + potential evaluation per
    line-search trial) continued from phi until budget_s seconds have passed.
    Returns the new phi and the sample's record; the sample covers
    evaluations / evals_per_step of a step of the workload.  cores is the
    process CPU time over the wall time (the oracle's FD integrals run on
    OpenMP threads, its FFTs on one)."""
    import resource
    import oracle as O
    r0 = resource.getrusage(resource.RUSAGE_SELF)
    t0 = time.perf_counter()
    n = iters = 0
    while True:
        if args.workload.startswith("eval"):
            O.evaluate(so, phi)
            n += 1
        else:
            phi, _, st = O.minimize(so, phi, gtol=1e-8, maxit=1)
            n += st["evaluations"]
            iters += max(st["iterations"], 1)
        if time.perf_counter() - t0 > budget_s:
            break
    dt = time.perf_counter() - t0
    r1 = resource.getrusage(resource.RUSAGE_SELF)
    cpu = (r1.ru_utime - r0.ru_utime) + (r1.ru_stime - r0.ru_stime)
    return phi, {"evaluations": n, "iterations": iters, "seconds": dt, "fraction": n / evals_per_step,
                 "cores": cpu / dt}


def cpu_baseline(args, evals_per_step, budget_s=15.0):
    """The oracle timed on a bounded sample of the workload (its own CG at
    full size for about budget_s seconds), converted to the workload's
    metric with the CG evaluations per step."""
    so, cfg, unit = oracle_system(args)
    import oracle as O
    phi = so.uniform_phi()
    O.evaluate(so, phi)                                             # warm-up (threads, caches)
    phi, rec = oracle_sample(args, so, phi, evals_per_step, budget_s)
    eps = rec["evaluations"] / rec["seconds"]
    return {"value": eps / evals_per_step, "unit": unit, "cores": int(round(rec["cores"])),
            "cores_measured": rec["cores"], "kind": "oracle",
            "sample": "the oracle's CG on the full-size (%s) workload: %d iterations, %d energy+potential "
                      "evaluations in %.1f s = %.3f evals/s, over %.1f evaluations per step; cores = "
                      "process CPU time / wall time" % ("x".join(map(str, cfg["grid"])), rec["iterations"],
                                                        rec["evaluations"], rec["seconds"], eps, evals_per_step)}


def run_reference(args):
    """Reference arm: the FP64 CPU oracle.  Each step is a bounded sample of
    the workload, about 4 s of the oracle's own CG at full size (a fraction
    of one MD step or solve: its evaluations over the evaluations a step
    takes); value = the steps' fractions over their measured time, so
    ms_per_step is the time actually timed per sample."""
    wl = WORKLOADS[args.workload]
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return None
    if wl["kind"] in ("batch", "serve"):
        return {"impl": "reference", "unavailable": "the oracle is timed on the md, solve and eval "
                "workloads; the batched and serving forms are GPU-only and carry their own "
                "sequential FP64 reference"}
    eps_step = EVALS_PER_STEP[args.workload]
    so, cfg, unit = oracle_system(args)
    import oracle as O
    phi = so.uniform_phi()
    for _ in range(args.warmup):
        O.evaluate(so, phi)
    recs = []
    for _ in range(args.steps):
        phi, rec = oracle_sample(args, so, phi, eps_step, 4.0)
        recs.append(rec)
    t = sum(r["seconds"] for r in recs)
    frac = sum(r["fraction"] for r in recs)
    nev = sum(r["evaluations"] for r in recs)
    value = frac / t
    cores = sum(r["cores"] * r["seconds"] for r in recs) / t
    metric, unit, conf = workload_meta(args.workload)
    conf["parallelism"] = "single process (host cores)"
    sample = ("each step: about 4 s of the oracle's CG on the full-size (%s) workload; %d evaluations "
              "in %.1f s over %d steps = %.3f evals/s, over %.1f evaluations per %s"
              % ("x".join(map(str, cfg["grid"])), nev, t, len(recs), nev / t, eps_step,
                 "MD step" if wl["kind"] == "md" else "solve"))
    return {"impl": "reference", "metric": metric, "value": value, "unit": unit,
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * t / len(recs), "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64 (binary64 throughout)", "data": "synthetic",
            "config": conf, "step_fraction": frac / len(recs),
            "cpu_baseline": {"value": value, "unit": unit, "cores": int(round(cores)),
                             "cores_measured": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": unit, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}


def main():
    args = parse()
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if args.impl == "reference":
        res = run_reference(args)
        if res is not None:
            print(json.dumps(res), flush=True)
        return
    if world > 1:
        import torch
        torch.distributed.init_process_group("nccl")
    kind = WORKLOADS[args.workload]["kind"]
    if kind == "eval":
        args.no_cpu = True
        res, eps = run_eval(args, rank, world)
    elif kind == "solve":
        res, eps = run_solve(args, rank, world)
    elif kind in ("batch", "serve"):
        args.no_cpu = True
        res, eps = (run_batch if kind == "batch" else run_serve)(args, rank, world)
    else:
        res, eps = run_ours(args, rank, world)
    if rank == 0:
        if not args.no_cpu:
            res["cpu_baseline"] = cpu_baseline(args, eps)
        print(json.dumps(res), flush=True)
    if world > 1:
        import torch
        torch.distributed.barrier()
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()
