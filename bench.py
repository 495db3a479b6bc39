#!/usr/bin/env python
"""Throughput benchmark of the matrix-valued quantum LBM step on GB300.

Default workload: D3Q19 128^3 periodic, tau = 0.7, beta0 = 1, density,
velocity (|u| <= 0.05) and spin fields as seeded Fourier-mode sums with
|k| <= 4, equilibrium-initialised (the 3D FP64/FP32 configuration).  One
"step" is one time step of the whole forward path: the fused
moments + equilibrium + BGK + in-place streaming kernel; the timed region
ends with the FP64 conservation reduction.  Reported:

  value       MLUPS of the FP32-storage step (sites x steps / s / 1e6)
  roofline    the step kernel's algorithmic bytes (b*4 values read + written
              per site) / its CUDA-event duration, against the measured HBM
              copy bandwidth
  fp16dev, fp64, fp64df, df64
              the same workload in the other storage precisions (FP16
              deviations; FP64; FP64 stepped in double-float arithmetic;
              double-float storage), each with its own roofline and clocks
  d2q9_4096   the D2Q9 4096^2 double shear layer, FP32 and FP16-deviation
  d3q19_512   the D3Q19 512^3 workload (41 GB FP32 state, tau = 0.6), fields
              synthesised on the device; MLUPS, GB/s and conservation drift
  e2e         MLUPS through the C ABI with host buffers: init from pinned
              host fields, K steps, moments back to pinned host memory
  adjoint     reverse sweep time (segment recomputation + adjoint steps) /
              plain forward time over the same steps, FP32: the D3Q19
              192^3 x 2000-step workload with square-root checkpoints (the
              quoted ratio), and the default workload over 256 steps with
              every state kept and with square-root checkpoints
  fd_params   the Fermi-Dirac parameter recovery (FP64 sweep, FD-path step,
              FP32 step with the fused single-precision solve)
  cpu_baseline  the FP64 oracle on a 32^3 sample on the host cores

Every leg after the first times at least --leg-ms of steps so that the
nvidia-smi clock samples fall inside its timed region.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
Under torchrun (N > 1) every rank runs an independent replica (no halo
exchange between ranks is implemented); value = all ranks' site updates /
max time.
"""
import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "MLUPS and % of HBM roofline (FP64 vs FP32 storage), adjoint/forward time ratio"

WORKLOADS = {
    "d3q19-128": dict(d=3, dims=(128, 128, 128), tau=0.7, beta0=1.0, kind="modes", seed=2,
                      desc="D3Q19 128^3 periodic, tau=0.7, beta0=1, Fourier-mode density/velocity/spin "
                           "fields |k|<=4 (RMS 0.02, |u|<=0.05), equilibrium init, eps=eps0"),
    "d2q9-64": dict(d=2, dims=(64, 64, 1), tau=0.8, beta0=1.0, kind="blob", seed=1,
                    desc="D2Q9 64^2 periodic, tau=0.8, beta0=1, density 1+0.05 sin(2 pi x/64), Gaussian "
                         "spin blob sigma=8 (|r|=0.1 n, seeded Bloch axis), u=0, eps=eps0"),
    "d3q19-512": dict(d=3, dims=(512, 512, 512), tau=0.6, beta0=1.0, kind="modes", seed=5,
                      desc="D3Q19 512^3 periodic, tau=0.6, beta0=1, Fourier-mode fields amplitude 0.02"),
    "d2q9-4096": dict(d=2, dims=(4096, 4096, 1), tau=0.7, beta0=1.0, kind="shear", seed=3,
                      desc="D2Q9 4096^2 periodic double shear layer, opposite spin bands"),
}


def bytes_per_value(prec):
    return {"fp64": 8, "df64": 8, "fp64df": 8, "fp32": 4, "fp16dev": 2}[prec]


def make_fields(w):
    from paper_1309_1656_gb300 import fields
    if w["kind"] == "modes":
        return fields.modes(w["d"], w["dims"], seed=w["seed"])
    if w["kind"] == "shear":
        return fields.shear2d(w["dims"][0], w["dims"][1], seed=w["seed"])
    if w["kind"] == "blob":
        return fields.blob2d(w["dims"][0], w["dims"][1], seed=w["seed"])
    raise ValueError(w["kind"])


STEP_KERNEL_SOURCES = ("lattice.cuh", "step.cuh")


def kernel_source_hash(files=STEP_KERNEL_SOURCES):
    """Hash of the sources that define the step kernel (collision + AA
    addressing); a recorded DRAM traffic is used only while it matches."""
    h = hashlib.sha256()
    for name in files:
        with open(os.path.join(ROOT, "paper_1309_1656_gb300", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def recorded_traffic(kernel_key):
    """DRAM bytes per site of a kernel from the committed ncu summary, if it
    was taken on the current kernel sources."""
    p = os.path.join(ROOT, "profiles", "ncu_traffic.json")
    if not os.path.exists(p):
        return None
    with open(p) as f:
        d = json.load(f)
    e = d.get(kernel_key)
    if not e or e.get("source_hash") != kernel_source_hash(tuple(e.get("hashed_files", STEP_KERNEL_SOURCES))):
        return None
    return float(e["dram_bytes_per_site"])


class ClockSampler:
    """nvidia-smi clocks and throttle reasons, sampled every 200 ms."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, dev_id):
        self.path = tempfile.mktemp(suffix=".csv")
        self.proc = None
        try:
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", dev_id, "--query-gpu=" + self.FIELDS,
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=self.f, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
        # wait (at most 3 s) until the sampler is running, so that it covers
        # the timed region that follows
        t0 = time.time()
        while self.proc is not None and time.time() - t0 < 3.0:
            if self.proc.poll() is not None:
                break
            self.f.flush()
            if os.path.getsize(self.path) > 0:
                break
            time.sleep(0.02)

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.f.close()
        rows = []
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) != 7:
                    continue
                try:
                    rows.append((float(parts[0]), float(parts[1]), parts[3:]))
                except ValueError:
                    continue
        os.unlink(self.path)
        if not rows:
            return None
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for _, _, r in rows for i, v in enumerate(r) if v.lower() == "active"})
        return {"sm_mhz": statistics.median(r[0] for r in rows), "sm_max_mhz": max(r[1] for r in rows),
                "reasons": reasons, "samples": len(rows)}


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def time_steps(lat, K, W, stream, torch, min_ms=0.0, ws=1):
    """W warm-up steps, then the timed region: Kt steps + the conservation
    reduction, CUDA events on the handle's stream.  Kt = K, or more when
    min_ms asks for a region long enough for the clock sampler (the per-step
    time is estimated from 4 extra warm-up steps).  Returns a dict."""
    lat.step(W)
    lat.sync()
    torch.cuda.synchronize()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    Kt = K
    if min_ms > 0:
        ev[0].record(stream)
        lat.step(4)
        ev[1].record(stream)
        torch.cuda.synchronize()
        est = max(ev[0].elapsed_time(ev[1]) / 4, 1e-4)
        Kt = max(K, 2 * int(np.ceil(min_ms / est / 2)))
        Kt = int(max_over_ranks_of(Kt, ws, "cuda"))
    ev[0].record(stream)
    lat.step(Kt)
    ev[1].record(stream)
    cons = lat.conserved()
    ev[2].record(stream)
    torch.cuda.synchronize()
    return dict(steps=Kt, step_ms=ev[0].elapsed_time(ev[1]) / Kt, total_ms=ev[0].elapsed_time(ev[2]), cons=cons)


def max_over_ranks_of(x, ws, device):
    """The largest of every rank's x (the job's time is its slowest rank's)."""
    if ws == 1:
        return x
    import torch
    t = torch.tensor([x], dtype=torch.float64, device=device)
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return float(t.item())


def job_mlups(ws, sites_per_rank, steps, seconds):
    """Whole-job throughput: all ranks' site updates over the slowest time."""
    return ws * sites_per_rank * steps / seconds / 1e6


# Step kernel per precision, and what bounds it when it is not HBM bandwidth.
STEP_KERNEL = {"fp32": "k_step_aa<%d, CodecF32>", "fp16dev": "k_step_aa_rows<%d, CodecF16Dev>",
               "fp64": "k_step_fix<%d>", "fp64df": "k_step_fix<%d>", "df64": "k_step_aa_df2<%d>"}
STEP_LIMIT = {"fp64": "issue: 1360 instructions per warp of 8 sites (fixed-point products, alignment); 57 % of "
                      "issue slots, integer pipe 62 %, multiply pipe 60 %, conversions 51 % busy",
              "fp64df": "issue: the FP64 kernel"}


class Bench:
    """Shared state of one bench run: device, stream, peaks, ranks."""

    def __init__(self, torch, qlbm, ws, rank, K, W):
        self.torch, self.qlbm, self.ws, self.rank, self.K, self.W = torch, qlbm, ws, rank, K, W
        self.peak, self.peak_src = measured_peaks()
        dev = torch.cuda.current_device()
        self.stream = torch.cuda.Stream()
        props = torch.cuda.get_device_properties(dev)
        uuid = str(getattr(props, "uuid", "")) or str(dev)
        self.dev_id = uuid if uuid.startswith("GPU-") else ("GPU-" + uuid if len(uuid) > 30 else str(dev))

    def barrier(self):
        if self.ws > 1:
            self.torch.distributed.barrier()

    def max_over_ranks(self, x):
        return max_over_ranks_of(x, self.ws, "cuda")

    def lattice(self, d, dims, tau, beta0, prec):
        return self.qlbm.Lattice(d, dims, tau, beta0, precision=prec, stream=self.stream.cuda_stream)

    def leg(self, d, dims, tau, beta0, prec, init, min_ms=0.0, clocks=True, traffic_key=None, extra_bytes=0):
        """One storage precision on one workload: init(lat) sets the state;
        then warm-up, the timed region (clocks sampled during it) and the
        conservation drift over it.  Returns the leg's record."""
        torch = self.torch
        N = dims[0] * dims[1] * dims[2]
        b = 9 if d == 2 else 19
        lat = self.lattice(d, dims, tau, beta0, prec)
        init(lat)
        c0 = lat.conserved()
        neg0 = self.qlbm.qlbm_negative_eq_count(lat.h)
        self.barrier()
        sampler = ClockSampler(self.dev_id) if clocks else None
        r = time_steps(lat, self.K, self.W, self.stream, torch, min_ms, self.ws)
        clk = sampler.stop() if sampler is not None else None
        neg1 = self.qlbm.qlbm_negative_eq_count(lat.h)
        lat.close()
        del lat
        torch.cuda.synchronize()
        step_ms = self.max_over_ranks(r["step_ms"])
        total_ms = self.max_over_ranks(r["total_ms"])
        alg = N * (b * 4 * 2 * bytes_per_value(prec) + extra_bytes)
        achieved = alg / (step_ms * 1e-3) / 1e9
        c1 = r["cons"]
        drift = float(np.max(np.abs(c1 - c0)) / np.max(np.abs(c0)))
        tb = recorded_traffic(traffic_key) if traffic_key else None
        roof = {"bound": "hbm", "achieved": round(achieved, 1), "peak": self.peak, "unit": "GB/s",
                "frac": round(achieved / self.peak, 4), "peak_source": self.peak_src,
                "traffic": None if tb is None else round(tb * N),
                "algorithmic_bytes_per_launch": alg, "kernel": STEP_KERNEL[prec] % d}
        if tb is not None:
            dram = tb * N / (step_ms * 1e-3) / 1e9
            roof["dram_achieved"] = round(dram, 1)
            roof["dram_frac"] = round(dram / self.peak, 4)
        if prec in STEP_LIMIT:
            roof["limit"] = STEP_LIMIT[prec]
        out = {"value": round(job_mlups(self.ws, N, r["steps"], total_ms * 1e-3), 1), "unit": "MLUPS",
               "steps": r["steps"], "ms_per_step": round(total_ms / r["steps"], 5),
               "kernel_mlups": round(job_mlups(self.ws, N, 1, step_ms * 1e-3), 1),
               "roofline": roof, "conservation_drift_rel": drift,
               "negative_eq_pairs": {"initial": neg0, "final": neg1, "of": N * b,
                                     "note": "(site, direction) pairs whose W_i^eq has a negative eigenvalue, "
                                             "before and after the timed steps (never clipped)"}}
        if clk:
            out["clocks"] = clk
        out["_step_ms"], out["_total_ms"] = step_ms, total_ms
        return out

    def adjoint(self, d, dims, tau, beta0, fl, NA, interval, box):
        """Plain forward, recording rollout and reverse sweep over NA FP32
        steps with checkpoint interval `interval` (0: the library's choice);
        observable: total s_z over the box (slices per axis)."""
        torch, qlbm, stream = self.torch, self.qlbm, self.stream
        N = dims[0] * dims[1] * dims[2]
        b = 9 if d == 2 else 19
        lat = self.lattice(d, dims, tau, beta0, "fp32")
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(6)]
        # the plain forward, timed twice (the faster counts: the first run
        # after large allocations and frees can be slowed by the device)
        t_plain = float("inf")
        for _ in range(2):
            lat.init_equilibrium(fl["rho4"], fl["u"], fl["eps"])
            lat.step(self.W)
            lat.sync()
            ev[0].record(stream)
            lat.step(NA)
            ev[1].record(stream)
            lat.sync()
            t_plain = min(t_plain, ev[0].elapsed_time(ev[1]))
        # an untimed rollout first allocates the checkpoint memory
        lat.init_equilibrium(fl["rho4"], fl["u"], fl["eps"])
        qlbm.qlbm_rollout(lat.h, NA, interval)
        lat.init_equilibrium(fl["rho4"], fl["u"], fl["eps"])
        torch.cuda.synchronize()
        ev[2].record(stream)
        qlbm.qlbm_rollout(lat.h, NA, interval)
        ev[3].record(stream)
        used = qlbm.qlbm_rollout_interval(lat.h)
        lam_T = torch.zeros((b, 4, N), dtype=torch.float64, device="cuda")
        grid = np.zeros(dims[::-1], bool)
        grid[box[::-1]] = True
        lam_T[:, 3, torch.from_numpy(grid.ravel()).cuda()] = 1.0
        lam_0 = torch.empty_like(lam_T)
        torch.cuda.synchronize()
        ev[4].record(stream)
        dJdtau = qlbm.qlbm_rollout_adjoint(lat.h, lam_T, lam_0)
        ev[5].record(stream)
        torch.cuda.synchronize()
        t_plain = self.max_over_ranks(t_plain)
        t_roll = self.max_over_ranks(ev[2].elapsed_time(ev[3]))
        t_adj = self.max_over_ranks(ev[4].elapsed_time(ev[5]))
        lat.close()
        del lat, lam_T, lam_0
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return {"ratio": round(t_adj / t_plain, 3), "interval": used, "steps": NA,
                "forward_ms": round(t_plain, 3), "rollout_ms": round(t_roll, 3), "adjoint_ms": round(t_adj, 3),
                "rollout_overhead": round(t_roll / t_plain, 3),
                "rollout_plus_sweep_over_forward": round((t_roll + t_adj) / t_plain, 3), "dJ_dtau": dJdtau}


def bench_ours(args):
    import torch
    ws, rank, local = dist_env()
    if ws > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    else:
        torch.cuda.set_device(0)
    import __graft_entry__
    from paper_1309_1656_gb300 import _build
    if not _build.up_to_date():
        if rank == 0:
            __graft_entry__.build()
        if ws > 1:
            torch.distributed.barrier()
    from paper_1309_1656_gb300 import fields, qlbm

    w = WORKLOADS[args.workload]
    d, dims = w["d"], w["dims"]
    N = dims[0] * dims[1] * dims[2]
    b = 9 if d == 2 else 19
    K, W = args.steps, args.warmup
    fl = make_fields(w)
    bn = Bench(torch, qlbm, ws, rank, K, W)
    stream = bn.stream
    peak = bn.peak

    def init_from(f):
        return lambda lat: lat.init_equilibrium(f["rho4"], f["u"], f["eps"])

    # the workload in every storage precision; the first is the line's value
    precs = args.precisions.split(",")
    prim = precs[0]
    results = {}
    for i, prec in enumerate(precs):
        results[prec] = bn.leg(d, dims, w["tau"], w["beta0"], prec, init_from(fl),
                               min_ms=0.0 if i == 0 else args.leg_ms,
                               traffic_key="step_%s_d%d" % (prec, d))

    extra = {}
    # the FP32 step with a magnetic field B(x) per site (Sec. 5): one unit
    # quaternion (16 B) read per site on top of the populations
    if "fp32" in results and d == 3 and not args.no_extra_workloads:
        nx, ny, nz = dims
        s_ = np.arange(N)
        x_, y_, z_ = s_ % nx, (s_ // nx) % ny, s_ // (nx * ny)
        Bs = np.array([0.05 + 0.04 * np.sin(2 * np.pi * x_ / nx), 0.03 * np.cos(2 * np.pi * y_ / ny),
                       0.08 + 0.05 * np.sin(2 * np.pi * z_ / nz + 1.0)])

        def init_field(lat):
            lat.set_magnetic_field_array(0.3, Bs)
            lat.init_equilibrium(fl["rho4"], fl["u"], fl["eps"])

        r = bn.leg(d, dims, w["tau"], w["beta0"], "fp32", init_field, min_ms=args.leg_ms, extra_bytes=16)
        r["field"] = "B(x) per site, mu = 0.3, smooth (|B| ~ 0.1); 608 + 16 algorithmic bytes per site"
        r["roofline"]["kernel"] = "k_step_aa<%d, CodecF32> (per-site field variant)" % d
        r["vs_no_field"] = round(r["_step_ms"] / results["fp32"]["_step_ms"], 3)
        extra["fp32_site_field"] = r
        del Bs

    # the other workloads: D2Q9 4096^2 shear layer (FP32, FP16-deviation)
    # and D3Q19 512^3 (FP32), fields synthesised on the device
    if not args.no_extra_workloads:
        w2 = WORKLOADS["d2q9-4096"]
        f2 = make_fields(w2)
        sub = {"workload": w2["desc"], "dims": list(w2["dims"]), "tau": w2["tau"]}
        for prec in ("fp32", "fp16dev"):
            sub[prec] = bn.leg(2, w2["dims"], w2["tau"], w2["beta0"], prec, init_from(f2), min_ms=args.leg_ms,
                               traffic_key="step_%s_d2_4096" % prec)
        extra["d2q9_4096"] = sub
        del f2
        w5 = WORKLOADS["d3q19-512"]
        spec = fields.mode_spec(3, w5["dims"], seed=w5["seed"])
        f5 = qlbm.fields_on_device(spec, w5["dims"], stream.cuda_stream)
        torch.cuda.synchronize()
        sub = {"workload": w5["desc"] + " (fields synthesised on the device by qlbm_fourier_field)",
               "dims": list(w5["dims"]), "tau": w5["tau"]}
        sub["fp32"] = bn.leg(3, w5["dims"], w5["tau"], w5["beta0"], "fp32", init_from(f5), min_ms=args.leg_ms,
                             traffic_key="step_fp32_d3_512")
        extra["d3q19_512"] = sub
        del f5
        torch.cuda.synchronize()
        torch.cuda.empty_cache()

    # reverse mode: the 192^3 x 2000-step workload with square-root
    # checkpoints (the one quoted against the <= 3x target), and the default
    # workload over 256 steps both with every state kept and with sqrt(N)
    # checkpoints
    adj = None
    if args.adjoint_steps > 0:
        c = lambda n: slice(n // 2 - max(1, n // 8), n // 2 + max(1, n // 8))
        box = tuple(c(n) for n in dims)
        NA = args.adjoint_steps
        ksq = int(np.ceil(np.sqrt(NA)))
        keep = bn.adjoint(d, dims, w["tau"], w["beta0"], fl, NA, 1, box)
        sq = bn.adjoint(d, dims, w["tau"], w["beta0"], fl, NA, ksq, box)
        adj = {"unit": "reverse sweep time / plain forward time, same steps",
               "observable": "total s_z over a central box", "precision": "fp32"}
        if args.adjoint_big_steps > 0:
            Lb = 192
            dimb = (Lb, Lb, Lb)
            fb = qlbm.fields_on_device(fields.mode_spec(3, dimb, seed=2), dimb, stream.cuda_stream)
            torch.cuda.synchronize()
            big = bn.adjoint(3, dimb, 0.7, 1.0, fb, args.adjoint_big_steps, 0,
                             tuple(slice(Lb // 2 - 16, Lb // 2 + 16) for _ in range(3)))
            del fb
            torch.cuda.empty_cache()
            big["workload"] = ("D3Q19 192^3, tau=0.7, FP32, Fourier-mode fields, %d steps, interval chosen by the "
                               "library (square-root checkpoints: the states do not fit), observable s_z over the "
                               "central 32^3 box" % args.adjoint_big_steps)
            adj["ratio"] = big["ratio"]
            adj["quoted"] = "sqrt(N) checkpoints on D3Q19 192^3 x %d steps" % args.adjoint_big_steps
            adj["sqrt_checkpoints_192"] = big
        else:
            adj["ratio"] = sq["ratio"]
            adj["quoted"] = "sqrt(N) checkpoints on the default workload"
        keep["note"] = "every state kept (written by the forward steps themselves); the sweep recomputes nothing"
        sq["note"] = "segment recomputation (two-buffer forward) + reverse steps"
        sq["dJ_dtau_matches_all_states_kept"] = sq["dJ_dtau"] == keep["dJ_dtau"]
        adj["sqrt_checkpoints"] = sq
        adj["all_states_kept"] = keep

    # Fermi-Dirac parameter recovery (side output, FP64 solve) and the FP64
    # step variant whose equilibrium goes through the recovered parameters
    fdp = None
    if args.fd_params and rank == 0:
        lat = bn.lattice(d, dims, w["tau"], w["beta0"], "fp64")
        lat.init_equilibrium(fl["rho4"], fl["u"], fl["eps"])
        lat.step(4)
        outs = [torch.empty((N,), dtype=torch.float64, device="cuda") for _ in range(3)]
        ax = torch.empty((3, N), dtype=torch.float64, device="cuda")
        qlbm.qlbm_fd_params(lat.h, *outs, ax)
        torch.cuda.synchronize()
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
        ev[0].record(stream)
        nfail = qlbm.qlbm_fd_params(lat.h, *outs, ax)
        ev[1].record(stream)
        lat.set_equilibrium_path(qlbm.QLBM_EQ_FD_PARAMS)
        ns = 10
        lat.step(2)
        lat.sync()
        ev[2].record(stream)
        lat.step(ns)
        ev[3].record(stream)
        torch.cuda.synchronize()
        t_fd = ev[0].elapsed_time(ev[1])
        t_step = ev[2].elapsed_time(ev[3]) / ns
        fdp = {"fd_params_ms": round(t_fd, 3), "fd_params_msites_per_s": round(N / t_fd / 1e3, 1),
               "fd_path_step_ms": round(t_step, 3), "fd_path_mlups": round(N / t_step / 1e3, 1),
               "unresolved_sites": nfail, "beta_median": float(outs[0].median()),
               "note": "FP64 per-site eigen-decomposition + Newton on the 3x3 logarithmic system (Prop. 1); cost reported "
                       "separately, the paper's step does not need it"}
        lat.close()
        del outs, ax
        torch.cuda.synchronize()
        # the FP32 step with the single-precision solve fused in: every step
        # also writes (beta, mu_up, mu_dn, axis) as float [6][N]
        if "fp32" in results:
            lat = bn.lattice(d, dims, w["tau"], w["beta0"], "fp32")
            lat.init_equilibrium(fl["rho4"], fl["u"], fl["eps"])
            o32 = [torch.empty((N,), dtype=torch.float32, device="cuda") for _ in range(3)]
            a32 = torch.empty((3, N), dtype=torch.float32, device="cuda")
            for _ in range(W):
                qlbm.qlbm_step_fd_output(lat.h, *o32, a32, count=False)
            lat.sync()
            torch.cuda.synchronize()
            nf = 100
            ev[0].record(stream)
            for _ in range(nf):
                qlbm.qlbm_step_fd_output(lat.h, *o32, a32, count=False)
            ev[1].record(stream)
            torch.cuda.synchronize()
            t_f = ev[0].elapsed_time(ev[1]) / nf
            nfail32 = qlbm.qlbm_step_fd_output(lat.h, *o32, a32)
            fbytes = N * (b * 4 * 2 * 4 + 6 * 4)
            fdp["fused_fp32"] = {
                "step_ms": round(t_f, 4), "mlups": round(N / t_f / 1e3, 1),
                "vs_plain_step": round(t_f / results["fp32"]["_step_ms"], 3),
                "achieved_gbs": round(fbytes / (t_f * 1e-3) / 1e9, 1),
                "hbm_frac": round(fbytes / (t_f * 1e-3) / 1e9 / peak, 4),
                "bytes_per_site": b * 4 * 2 * 4 + 6 * 4, "unresolved_sites": nfail32,
                "note": "FP32 step + per-site single-precision FD solve (double where the float "
                        "iteration does not settle), parameters written every step"}
            lat.close()
            del o32, a32
            torch.cuda.synchronize()

    # end-to-end through the C ABI with pinned host buffers
    e2e = None
    if not args.no_e2e:
        pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()
        r4, uu = pin(fl["rho4"]), pin(fl["u"])
        out_r = torch.empty((4, N), dtype=torch.float64).pin_memory().numpy()
        out_u = torch.empty((d, N), dtype=torch.float64).pin_memory().numpy()
        out_e = torch.empty((N,), dtype=torch.float64).pin_memory().numpy()
        lat = bn.lattice(d, dims, w["tau"], w["beta0"], prim)
        lat.init_equilibrium(r4, uu)       # warm the staging buffers
        lat.step(W)
        qlbm.qlbm_moments(lat.h, out_r, out_u, out_e)
        bn.barrier()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        qlbm.qlbm_init_equilibrium(lat.h, r4, uu, None)
        qlbm.qlbm_step(lat.h, K)
        qlbm.qlbm_moments(lat.h, out_r, out_u, out_e)
        t1 = time.perf_counter()
        dt_e2e = bn.max_over_ranks(t1 - t0)
        lat.close()
        e2e = {"value": round(job_mlups(ws, N, K, dt_e2e), 3), "unit": "MLUPS",
               "h2d_bytes_per_step": (r4.nbytes + uu.nbytes) / K,
               "d2h_bytes_per_step": (out_r.nbytes + out_u.nbytes + out_e.nbytes) / K}

    growth = None
    if args.error_growth > 0 and rank == 0:
        growth = error_growth(w, fl, args.error_growth, args.error_every, torch, qlbm)

    if rank != 0:
        if ws > 1:
            torch.distributed.destroy_process_group()
        return

    def parity(sdims, sfl, nsteps, st_ref, mom_ref):
        """Errors of the GPU precisions against the oracle on the CPU sample
        (normwise, max |x - x_ref| / max |x_ref|)."""
        err = lambda a, b_: float(np.max(np.abs(a - b_)) / np.max(np.abs(b_)))
        res = {"steps": nsteps, "norm": "max |x - x_oracle| / max |x_oracle|"}
        for prec in ("fp64", "fp64df", "df64", "fp32", "fp16dev"):
            with qlbm.Lattice(d, sdims, w["tau"], w["beta0"], precision=prec) as lat:
                lat.init_equilibrium(sfl["rho4"], sfl["u"], sfl["eps"])
                lat.step(nsteps)
                r4, uu, ee = lat.moments()
                e = {"n": err(r4[0], mom_ref[0][0]), "S": err(r4[1:], mom_ref[0][1:]),
                     "u": err(uu, mom_ref[1]), "eps": err(ee, mom_ref[2])}
                if prec in ("fp64", "fp64df", "df64"):
                    e["state"] = err(lat.get_state(), st_ref)
                    e["state_per_step"] = e["state"] / nsteps
                res[prec] = {k: float("%.3g" % v) for k, v in e.items()}
        return res

    cpu = None
    if ws == 1 and not args.no_cpu:
        cpu = cpu_baseline(w, target_s=args.cpu_seconds, parity_fn=parity)

    def public(r):
        return {k: v for k, v in r.items() if not k.startswith("_")}

    r0 = results[prim]
    line = {
        "metric": METRIC, "value": round(job_mlups(ws, N, K, r0["_total_ms"] * 1e-3), 1), "unit": "MLUPS",
        "n_gpus": ws, "steps": K, "warmup": W, "ms_per_step": round(r0["_total_ms"] / K, 5),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": {"fp32": "f32", "fp64": "f64", "fp16dev": "f16-storage/f32", "df64": "f32x2",
                  "fp64df": "f64-storage/f32x2"}[prim],
        "data": "synthetic",
        "config": {"workload": w["desc"], "lattice": "D3Q19" if d == 3 else "D2Q9",
                   "dims": list(dims), "sites": N, "tau": w["tau"], "beta0": w["beta0"],
                   "precision": prim, "parallelism": "replicas" if ws > 1 else "single-gpu",
                   "l2": ("inputs larger than L2: state %.2f GB > 129 MB, no flush" if
                          N * b * 4 * bytes_per_value(prim) > 129e6 else
                          "state %.4f GB fits in the 129 MB L2: L2-resident by construction, "
                          "not an HBM measurement") % (N * b * 4 * bytes_per_value(prim) / 1e9)},
        "roofline": r0["roofline"],
        "kernel_mlups": r0["kernel_mlups"],
        "conservation_drift_rel": r0["conservation_drift_rel"],
        "gpu_launches": K + 2,
    }
    if "clocks" in r0:
        line["clocks"] = r0["clocks"]
    for p_, r in results.items():
        if p_ != prim:
            line[p_] = public(r)
    for k_, sub in extra.items():
        line[k_] = {k: (public(v) if isinstance(v, dict) and not k.startswith("_") else v)
                    for k, v in sub.items() if not k.startswith("_")}
    if growth:
        line["error_growth"] = growth
    if e2e:
        line["e2e"] = e2e
    if adj:
        line["adjoint"] = adj
    if fdp:
        line["fd_params"] = fdp
    if cpu:
        line["cpu_baseline"] = cpu
    print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()


def error_growth(w, fl, total, every, torch, qlbm):
    """Normwise errors of the double-float, FP32 and FP16-deviation moment
    fields against the FP64 run of the same workload, every `every` steps."""
    d, dims = w["d"], w["dims"]
    N = dims[0] * dims[1] * dims[2]
    lats = {p: qlbm.Lattice(d, dims, w["tau"], w["beta0"], precision=p) for p in ("fp64", "df64", "fp32", "fp16dev")}
    for lat in lats.values():
        lat.init_equilibrium(fl["rho4"], fl["u"], fl["eps"])
    bufs = {p: (torch.empty((4, N), dtype=torch.float64, device="cuda"),
                torch.empty((d, N), dtype=torch.float64, device="cuda"),
                torch.empty((N,), dtype=torch.float64, device="cuda")) for p in lats}
    out = []
    t = 0
    while t < total:
        n = min(every, total - t)
        for lat in lats.values():
            lat.step(n)
        t += n
        for p, lat in lats.items():
            qlbm.qlbm_moments(lat.h, *bufs[p])
        ref = bufs["fp64"]

        def err(a, b_):
            return float((a - b_).abs().max() / b_.abs().max())

        row = {"step": t}
        for p in ("df64", "fp32", "fp16dev"):
            r, u, e = bufs[p]
            row[p] = {"n": err(r[0], ref[0][0]), "S": err(r[1:], ref[0][1:]), "u": err(u, ref[1]),
                      "eps": err(e, ref[2])}
        out.append(row)
    for lat in lats.values():
        lat.close()
    return {"reference": "the FP64 GPU run of the same workload (itself within 1e-12/step of the oracle)",
            "norm": "max |x - x_fp64| / max |x_fp64| per field", "rows": out}


def cpu_sample(w, L=32):
    from paper_1309_1656_gb300 import fields
    d = w["d"]
    if w["kind"] == "blob":
        return w["dims"], make_fields(w)
    dims = (L, L, L) if d == 3 else (L * 8, L * 8, 1)
    fl = fields.modes(d, dims, seed=w["seed"]) if w["kind"] == "modes" else \
        fields.shear2d(dims[0], dims[1], seed=w["seed"], delta=max(2.0, 80.0 * dims[1] / 4096.0))
    return dims, fl


def cpu_baseline(w, target_s=15.0, parity_fn=None):
    """The FP64 oracle, as it stands, on a bounded sample of the workload.
    With parity_fn, the GPU precisions run the same sample for 1000 steps
    and report their error against the oracle's result."""
    import oracle
    oracle.build()
    d = w["d"]
    dims, fl = cpu_sample(w)
    N = dims[0] * dims[1] * dims[2]
    cores = oracle.max_threads(0)
    st = oracle.init_equilibrium(d, dims, w["beta0"], fl["rho4"], fl["u"], fl["eps"])
    st = oracle.run(d, dims, w["tau"], w["beta0"], 2, st)      # thread start-up
    # run in chunks until the sample has taken target_s of wall time
    n, chunk, dt = 0, 8, 0.0
    while dt < target_s:
        t = time.perf_counter()
        st = oracle.run(d, dims, w["tau"], w["beta0"], chunk, st)
        dt += time.perf_counter() - t
        n += chunk
        chunk = min(2 * chunk, 4096)
    out = {"value": round(N * n / dt / 1e6, 3), "unit": "MLUPS", "cores": cores, "kind": "oracle",
           "sample": "%s sub-lattice %s of the same workload recipe, %d FP64 steps, %.1f s" %
                     ("D3Q19" if d == 3 else "D2Q9", "x".join(map(str, dims)), n, dt)}
    # the same sample on one thread, over a shorter bounded time
    n1, chunk, dt1 = 0, 1, 0.0
    while dt1 < target_s / 4:
        t = time.perf_counter()
        st = oracle.run(d, dims, w["tau"], w["beta0"], chunk, st, nthreads=1)
        dt1 += time.perf_counter() - t
        n1 += chunk
        chunk = min(2 * chunk, 512)
    out["single_thread"] = {"value": round(N * n1 / dt1 / 1e6, 3), "unit": "MLUPS", "cores": 1,
                            "steps": n1, "seconds": round(dt1, 2)}
    if parity_fn is not None:   # 1000 steps: the fields have not yet relaxed away
        st = oracle.init_equilibrium(d, dims, w["beta0"], fl["rho4"], fl["u"], fl["eps"])
        st = oracle.run(d, dims, w["tau"], w["beta0"], 1000, st)
        out["parity"] = parity_fn(dims, fl, 1000, st, oracle.moments(d, dims, w["beta0"], st))
    return out


def bench_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return
    import oracle
    oracle.build()
    w = WORKLOADS[args.workload]
    d = w["d"]
    dims, fl = cpu_sample(w)
    N = dims[0] * dims[1] * dims[2]
    cores = oracle.max_threads(0)
    st = oracle.init_equilibrium(d, dims, w["beta0"], fl["rho4"], fl["u"], fl["eps"])
    st = oracle.run(d, dims, w["tau"], w["beta0"], args.warmup, st)
    t = time.perf_counter()
    oracle.run(d, dims, w["tau"], w["beta0"], args.steps, st)
    dt = time.perf_counter() - t
    v = N * args.steps / dt / 1e6
    line = {"impl": "reference", "metric": METRIC, "value": round(v, 3), "unit": "MLUPS",
            "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": round(dt * 1e3 / args.steps, 4), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": w["desc"], "sample": "x".join(map(str, dims)),
                       "note": "reference arm = the FP64 CPU oracle (no reference implementation exists)"},
            "cpu_baseline": {"value": round(v, 3), "unit": "MLUPS", "cores": cores, "kind": "oracle",
                             "sample": "%s sub-lattice %s per step" %
                                       ("D3Q19" if d == 3 else "D2Q9", "x".join(map(str, dims)))},
            "e2e": {"value": round(v, 3), "unit": "MLUPS", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=1000)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="d3q19-128", choices=sorted(WORKLOADS))
    ap.add_argument("--precisions", default="fp32,fp16dev,fp64,fp64df,df64",
                    help="storage precisions of the workload; the first gives the line's value")
    ap.add_argument("--leg-ms", type=float, default=600.0,
                    help="least timed-region length of every leg after the first (clock sampling)")
    ap.add_argument("--no-extra-workloads", action="store_true",
                    help="skip the D2Q9 4096^2 and D3Q19 512^3 legs")
    ap.add_argument("--adjoint-big-steps", type=int, default=2000,
                    help="steps of the D3Q19 192^3 reverse-mode leg (0: skip it)")
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--adjoint-steps", type=int, default=256)
    ap.add_argument("--error-growth", type=int, default=0,
                    help="also run FP64/FP32/FP16 side by side for this many steps and report errors")
    ap.add_argument("--error-every", type=int, default=1000)
    ap.add_argument("--no-fd-params", dest="fd_params", action="store_false",
                    help="skip timing the Fermi-Dirac parameter recovery")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        bench_reference(args)
    else:
        bench_ours(args)


if __name__ == "__main__":
    main()
