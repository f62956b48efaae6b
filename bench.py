"""Benchmark of the non-stationary Matern GP hot path on one GB300 per rank.

A step is one conjugate-gradient iteration on (K~ + eta^2 I) through the C ABI
(gp_cg_solve): the matvec (spread, forward FFT, step 3, inverse FFT, interp) plus
the float64 CG reductions and vector updates.  The metric is matvec throughput,
points x right-hand sides per second (Mpts/s), on the 2-D clustered workload
(N = 1e6: half uniform on the unit square, half in 8 Gaussian clusters, Matern
nu = 3/2, eps = 1e-6).  Default path: FP32 spread/FFT/step 3/interp with float64
CG; the plain float64 path is timed beside it.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Under torchrun each rank runs an independent replica (no collective on the data
path); rank 0 prints one JSON line with the max over ranks.
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

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = ("NUFFT matvec Mpts/s (one CG iteration on K~ + eta^2 I, float64-grade), 2-D clustered N=1e6, Matern 3/2, "
          "eps=1e-6")
UNIT = "Mpts/s"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=1_000_000)
    ap.add_argument("--nu", type=float, default=1.5)
    ap.add_argument("--eps", type=float, default=1e-6)
    ap.add_argument("--precision", default="df64", choices=["df64", "fp64", "fp32"],
                    help="arithmetic of the headline path: df64 float-float (float64-grade, the default), "
                         "fp64 native float64, fp32")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--side", action="store_true",
                    help="also run the side measurements (config 1 latency, batched R, config 2 at nu = 1/2, "
                         "config 3, served solves); each prints its wall time to stderr as it ends")
    ap.add_argument("--no-extras", action="store_true",
                    help="no side measurements (the default; kept so that recorded commands still run)")
    ap.add_argument("--serve-requests", type=int, default=12)
    ap.add_argument("--profile-case", action="store_true",
                    help="a fixed workload for profilers: build one plan (--d, --n, --eps, --precision, "
                         "--transform) and run --matvecs matvecs, nothing else")
    ap.add_argument("--solve-compare", action="store_true",
                    help="time to solution on the benchmark workload: plain float64-grade CG against the "
                         "refined FP32 solve, both to --rtol, and the difference of the two solutions")
    ap.add_argument("--rtol", type=float, default=1e-8)
    ap.add_argument("--d", type=int, default=2, choices=[2, 3])
    ap.add_argument("--matvecs", type=int, default=4)
    ap.add_argument("--transform", type=int, default=0)
    return ap.parse_args()


def job_totals(ms_total: float, points_per_step: float, ws: int, device=None):
    """Whole-job figures over the ranks: the slowest rank's elapsed milliseconds and the
    points all ranks processed per step (replicas may hold different N).  One rank: the
    arguments unchanged."""
    if ws <= 1:
        return float(ms_total), float(points_per_step)
    import torch
    import torch.distributed as dist
    t_ms = torch.tensor([float(ms_total)], dtype=torch.float64, device=device)
    t_pts = torch.tensor([float(points_per_step)], dtype=torch.float64, device=device)
    dist.all_reduce(t_ms, op=dist.ReduceOp.MAX)
    dist.all_reduce(t_pts, op=dist.ReduceOp.SUM)
    return float(t_ms.item()), float(t_pts.item())


def dist_setup():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


# ------------------------------------------------------------------ clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.idx = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.idx), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "of measured"
    return 6800.0, "of fallback"


# ------------------------------------------------------------------ workload
def workload(args):
    import gpinputs
    w = gpinputs.config_2d(args.n, args.nu)
    w.eps = args.eps
    return w


def own_columns(info):
    """Whether a 2-D plan's column transforms are the library's own (csrc/fft2d.cu, own_cols;
    0 float64, 1 FP32, 2 float-float).  For plans that hold their spare tables: the ones built here
    have no max_bytes."""
    if info["precision"] == 2:
        return True
    return 256 <= info["nf"] <= (4096 if info["precision"] == 1 else 8192)


def algorithmic_bytes(info, N, R, rs):
    """Algorithmic HBM bytes per launch of each matvec phase (reads + writes once).

    ext = the grid rows/columns that hold data (the point box on the fine grid plus one
    kernel width); cplx = 2 rs.  Transform 3 (d = 2): the row stages read/write ext^2
    real values and (M+1) ext modes per channel, the column transforms (M+1) nf complex
    each way, step 3 the mode box (M+1)(2M+1) plus A' on the quadrant (M+1)^2."""
    d, nf, M, W = info["d"], info["nf"], info["M"], info["kernel_width"]
    C = info["n_sigma"] + 1
    L = max(info["box_hi"][a] - info["box_lo"][a] for a in range(d))
    ext = min(nf, int(math.ceil(nf * info["dw"] * L)) + W)
    G, Gocc = nf ** d, ext ** d
    cp = 2 * rs
    pts = N * (d * (4 + rs) + C * rs + 4)          # l0, xi, w_k, bin pointers
    pairs = C * (C + 1) // 2
    out = {"spread": C * R * Gocc * rs + pts + N * R * 8, "interp": C * R * Gocc * rs + pts + 2 * N * R * 8}
    if info["transform"] == 3:
        rows = C * R * (Gocc * rs + (M + 1) * ext * cp)
        if own_columns(info):
            # the column kernels read the rows that can be nonzero and write the rows the
            # next stage reads: the data extent and the 2M + 1 kept modes
            cols = C * R * (M + 1) * (ext + 2 * M + 1) * cp
        else:
            cols = 2 * C * R * (M + 1) * nf * cp
        box = C * R * (M + 1) * (2 * M + 1) * cp
        out.update(fft_fwd=rows + cols, fft_inv=rows + cols, diag=2 * box + pairs * (M + 1) ** 2 * rs,
                   rows_fwd=rows, rows_inv=rows, cols_fwd=cols, cols_inv=cols)
    else:
        S = nf ** (d - 1) * (nf // 2 + 1)
        nfreq = (2 * M + 1) ** (d - 1) * (M + 1)
        out.update(fft_fwd=C * R * (G * rs + S * cp), fft_inv=C * R * (S * cp + G * rs),
                   diag=C * R * nfreq * cp + pairs * nfreq * rs + C * R * S * cp)
        # the 1-D row transforms (no cuFFT) do the whole phase
        out.update(rows_fwd=out["fft_fwd"], rows_inv=out["fft_inv"])
    return out


# DRAM bytes (dram__bytes_read.sum + dram__bytes_write.sum) per launch from one ncu capture of
# the current kernels on the 2-D clustered workload (N = 1e6, eps = 1e-6, FP32, transform 3):
# rows + column transform for the FFT phases.  (The library's kernels on the same cloud held to
# three standard deviations, M = 2802 where the workload's own plan has 2818.)  Reported as `traffic`
# only for that workload, and to be re-taken whenever these kernels change.
MEASURED_TRAFFIC = {
    ("d2_N1000000_clustered_matern32", "f32", 1e-06): {
        "spread": 0.061e9 + 1.103e9,
        "fft_fwd": (1.193e9 + 1.106e9) + (1.663e9 + 1.607e9),
        "diag": 2.553e9 + 1.100e9,
        "fft_inv": (1.663e9 + 1.607e9) + (1.151e9 + 1.115e9),
        "interp": 1.225e9 + 0.008e9,
        "rows_fwd": 1.193e9 + 1.106e9,
        "rows_inv": 1.151e9 + 1.115e9,
    },
}


PHASES = ["spread", "fft_fwd", "diag", "fft_inv", "interp"]


def launches_per_step(own_columns: bool) -> int:
    """Our kernels in one CG iteration on the 2-D path: spread, forward rows, step 3, inverse
    rows, interp, and the CG kernels (dot partial + final, update_xr + dot final, update_p,
    roll, check); the two column transforms are ours or cuFFT's (own_columns)."""
    return 5 + 7 + (2 if own_columns else 0)


# FP32 operations of the float-float arithmetic (ff64.h, fft_core.h) in the passes: a sum
# without the closing renormalisation 8 (TwoSum 6, low words 2), a product 7 (product, three
# fused multiply-adds, FastTwoSum 3), a normalised sum 11; complex: sum 16, product 34 (each
# component two TwoProds with cross terms, a TwoSum, two closing operations), renormalisation
# of a pass output 6.  In-register DFTs: DFT-2 32, DFT-4 128, DFT-8 456 (two DFT-4, the W8^1
# and W8^3 rotations at 36 each, eight complex sums), DFT-16 1376 (two DFT-8, four W16
# rotations as complex products, two W8 rotations, sixteen complex sums).  A radix-16
# Stockham pass with twiddles: DFT-16, 15 complex products and 16 renormalisations, 1982 per
# 16 points; a first pass at span 1 has no twiddles.
FF_DFT = {2: 32, 4: 128, 8: 456, 16: 1376}
FF_RENORM16 = 16 * 6
FF_PASS16 = 1376 + 15 * 34 + FF_RENORM16


def ff_fft_ops(L: int) -> int:
    """FP32 operations of one length-2^L complex FFT in the kernels' pass schedule: a first
    pass of radix 2^(L mod 4) (or 16) at span 1 without twiddles, then radix-16 passes."""
    r0 = 16 if L % 4 == 0 else 1 << (L % 4)
    passes = L // 4 - (1 if L % 4 == 0 else 0)
    nt = (1 << L) // 16
    return nt * ((16 // r0) * FF_DFT[r0] + FF_RENORM16 + passes * FF_PASS16)


def alu_ops(info, R):
    """FP32 operations per launch of the float-float transform kernels, counted from their
    arithmetic (the algorithm as emulated: the bound is the FP32 issue rate).
    rows_fwd: per grid row of the data extent an nf/2-point complex FFT, then per kept mode
      the real split (two complex sums, a complex product, two normalised sums and two
      halvings: 102) and the split twiddle (a complex product, shared by the RB rows of a
      block);
    rows_inv: the merge of each mode pair (per pair of the nf/2 + 1 modes two complex sums,
      one complex product, two normalised complex sums: 110, and one twiddle of 34), then the
      nf/2-point FFT;
    cols_*: one nf-point complex FFT per kept mode column."""
    nf, M, W = info["nf"], info["M"], info["kernel_width"]
    C = info["n_sigma"] + 1
    L = max(info["box_hi"][a] - info["box_lo"][a] for a in range(info["d"]))
    ext = min(nf, int(math.ceil(nf * info["dw"] * L)) + W)
    l2 = int(round(math.log2(nf // 2)))
    rows = C * R * ext
    fwd = rows * (ff_fft_ops(l2) + (M + 1) * 102) + C * R * (ext // 2) * (M + 1) * 34
    inv = rows * (ff_fft_ops(l2) + (nf // 4 + 1) * (110 + 34))
    cols = C * R * (M + 1) * ff_fft_ops(int(round(math.log2(nf))))
    return {"rows_fwd": fwd, "rows_inv": inv, "cols_fwd": cols, "cols_inv": cols}


# FP32 lanes x SMs x maximum SM clock (152 x 128 x 2.07 GHz): the issue ceiling of FP32
# instructions (a fused multiply-add is one), the peak of the float-float kernels
FP32_ISSUE_PEAK = 152 * 128 * 2.07e9


def roof_of(ab, name, ms, peak, peak_src, traffic, alu_ops=None):
    """The roofline entry of one kernel: HBM (algorithmic bytes / time against the measured
    copy rate), or, for the float-float transform kernels, the FP32 issue rate (their
    counted FP32 operations / time against FP32_ISSUE_PEAK), with the HBM figure beside it."""
    ach = ab[name] / (ms * 1e-3) / 1e9
    out = {"kernel": name, "bound": "hbm", "achieved": round(ach, 1), "peak": peak, "unit": "GB/s",
           "frac": round(ach / peak, 4), "peak_source": peak_src,
           "traffic": int(traffic) if traffic is not None else None,
           "algorithmic_bytes": int(ab[name]), "ms_per_launch": round(ms, 4)}
    if alu_ops:
        ops = alu_ops / (ms * 1e-3)
        out.update({"bound": "alu", "achieved": round(ops / 1e12, 3), "peak": round(FP32_ISSUE_PEAK / 1e12, 3),
                    "unit": "T FP32 op/s", "frac": round(ops / FP32_ISSUE_PEAK, 4),
                    "peak_source": "derived: 152 SMs x 128 FP32 lanes x 2.07 GHz",
                    "algorithmic_ops": int(alu_ops),
                    "hbm": {"achieved_gbs": round(ach, 1), "peak_gbs": peak, "frac": round(ach / peak, 4)}})
    return out


PRECISIONS = {"fp32": ("GP_FP32", "f32", 4, "f32 spread/FFT/step 3/interp, f64 CG reductions"),
              "fp64": ("GP_FP64", "f64", 8, "f64 throughout"),
              "df64": ("GP_DF64", "df64", 8, "float-float (two f32 words, about 48 significant bits) in spread, "
                                           "FFT, step 3 and interp on the FP32 pipe; f64 CG reductions")}


def _cg(abi, pl, k, yy, xx, eta2):
    st, it, rel = abi.gp_cg_solve(pl.handle, yy, xx, 1, eta2, 1e-30, k)
    return it[0]


def _timed_steps(abi, torch, pl, k, yy, xx, eta2, stream):
    """One event pair on the launching stream around exactly k CG iterations."""
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    it = _cg(abi, pl, k, yy, xx, eta2)
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1), it


def _step_distribution(abi, torch, pl, blocks, yy, xx, eta2, stream):
    """Per-step milliseconds from `blocks` separate one-iteration solves, each bracketed by
    its own events (median and p10/p90 of these)."""
    out = []
    for _ in range(blocks):
        ms, it = _timed_steps(abi, torch, pl, 1, yy, xx, eta2, stream)
        out.append(ms / max(it, 1))
    q = np.percentile(out, [10, 50, 90])
    return {"runs": blocks, "p10_ms": round(float(q[0]), 4), "median_ms": round(float(q[1]), 4),
            "p90_ms": round(float(q[2]), 4),
            "note": "each run one gp_cg_solve call of one iteration (includes its start-up: x0 = 0, r = y, "
                    "two dot products)"}


def _phases(abi, pl, y, x, eta2, k):
    """Per-phase and row-kernel milliseconds from the library's own events (a separate pass)."""
    abi.gp_profile_enable(pl.handle, True)
    _cg(abi, pl, k, y, x, eta2)
    phase_ms, n_rec = abi.gp_profile_read(pl.handle)
    rows_ms = abi.gp_profile_read_rows(pl.handle)
    abi.gp_profile_enable(pl.handle, False)
    return phase_ms, rows_ms, n_rec


def _kernel_ms(phase_ms, rows_ms, own_columns):
    """Our own kernels: spread, step 3, interp, the row kernels inside the transform phases,
    and (own_columns) the column kernels, the rest of those phases."""
    km = {"spread": phase_ms[0], "diag": phase_ms[2], "interp": phase_ms[4]}
    for name, ms in zip(("rows_fwd", "rows_inv"), rows_ms):
        if ms > 0:
            km[name] = ms
    if own_columns:
        km["cols_fwd"] = phase_ms[1] - rows_ms[0]
        km["cols_inv"] = phase_ms[3] - rows_ms[1]
    return km


def run_ours(args, ws, rank, local):
    import torch
    import paper_2407_03608_gb300 as gpn
    from paper_2407_03608_gb300 import abi
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    w = workload(args)
    N = w.N
    pname, dtype, rs, arith = PRECISIONS[args.precision]
    prec = getattr(gpn, pname)
    eta2 = w.eta ** 2
    pts = torch.from_numpy(w.points).to(dev)
    s = torch.from_numpy(w.s).to(dev)
    l = torch.from_numpy(w.l).to(dev)
    y = torch.from_numpy(w.y).to(dev)
    t0 = time.perf_counter()
    plan = gpn.Plan(pts, s, l, nu=w.nu, eps=w.eps, precision=prec)
    torch.cuda.synchronize()
    plan_s = time.perf_counter() - t0
    info = plan.info
    stream = torch.cuda.current_stream()
    x = torch.empty_like(y)

    # warm-up, then the timed region: K CG iterations, events on the launching stream
    _cg(abi, plan, max(args.warmup, 1), y, x, eta2)
    torch.cuda.synchronize()
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()
    ms_total, iters = _timed_steps(abi, torch, plan, args.steps, y, x, eta2, stream)
    if ws > 1:
        dist.barrier()
    clocks = sampler.stop()
    dist_stats = _step_distribution(abi, torch, plan, max(20, min(args.steps, 40)), y, x, eta2, stream)
    phase_ms, rows_ms, n_rec = _phases(abi, plan, y, x, eta2, min(args.steps, 10))
    ms_total, points_job = job_totals(ms_total, N, ws, dev)
    ms_step = ms_total / iters
    value = points_job / (ms_step * 1e-3) / 1e6

    # end to end through the public API with pinned host buffers: every step copies
    # y in and alpha out (gp_cg_solve with host pointers runs one iteration per call)
    yh = torch.from_numpy(w.y.copy()).pin_memory()
    xh = torch.empty_like(yh).pin_memory()
    e2e_steps = max(3, min(args.steps, 10))
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        abi.gp_cg_solve(plan.handle, yh, xh, 1, eta2, 1e-30, 1)
    e2e_s = (time.perf_counter() - t0) / e2e_steps
    e2e = {"value": ws * N / e2e_s / 1e6, "unit": UNIT, "h2d_bytes_per_step": 8 * N, "d2h_bytes_per_step": 8 * N,
           "ms_per_step": e2e_s * 1e3}

    a = torch.from_numpy(w.alpha).to(dev)
    out_main = plan.matvec(a)
    peak, peak_src = measured_peaks()
    extra = {}

    def err_pair(u, v):
        return {"rel_l2": float(torch.linalg.norm(u - v) / torch.linalg.norm(v)),
                "rel_max": float((u - v).abs().max() / v.abs().max())}

    def leg(pl, pn):
        """Another precision on the same K~: the same K steps, its kernels' rooflines."""
        xx = torch.empty_like(y)
        _cg(abi, pl, 2, y, xx, eta2)
        ms_k, it_k = _timed_steps(abi, torch, pl, args.steps, y, xx, eta2, stream)
        ph, rw, _ = _phases(abi, pl, y, xx, eta2, min(args.steps, 5))
        ab_k = algorithmic_bytes(pl.info, N, 1, PRECISIONS[pn][2])
        km = _kernel_ms(ph, rw, own_columns(pl.info))
        return {"value": round(N / (ms_k / it_k * 1e-3) / 1e6, 3), "ms_per_step": round(ms_k / it_k, 4),
                "steps": it_k, "arith": PRECISIONS[pn][3],
                "phase_ms": {PHASES[q]: round(ph[q], 4) for q in range(5)},
                "roofline_kernels": [roof_of(ab_k, k, v, peak, peak_src, None) for k, v in km.items()]}

    # the plain float64 GPU path on the same K~ (the comparison of the metric)
    if prec != gpn.GP_FP64:
        p64 = gpn.Plan(pts, s, l, nu=w.nu, eps=w.eps, precision=gpn.GP_FP64, **plan.matched_opts())
        o64 = p64.matvec(a)
        extra["matvec_err_vs_fp64_gpu"] = err_pair(out_main, o64)
        extra["fp64_path"] = leg(p64, "fp64")
    else:
        o64 = out_main
    # the mixed-precision FP32 path on the same K~
    if prec != gpn.GP_FP32:
        p32 = gpn.Plan(pts, s, l, nu=w.nu, eps=w.eps, precision=gpn.GP_FP32, **plan.matched_opts())
        m32 = leg(p32, "fp32")
        m32["matvec_err_vs_fp64_gpu"] = err_pair(p32.matvec(a), o64)
        extra["mixed_fp32"] = m32
        p32.close()
    if prec != gpn.GP_FP64:
        p64.close()
    out_sample = out_main.cpu().numpy()

    ab = algorithmic_bytes(info, N, 1, rs)
    kern_ms = _kernel_ms(phase_ms, rows_ms, own_columns(plan.info))
    dom = max(range(5), key=lambda q: phase_ms[q])
    dom_ours = max(kern_ms, key=kern_ms.get)
    traffic = MEASURED_TRAFFIC.get((w.name, dtype, w.eps), {})
    tr_ok = args.n == 1_000_000
    alu = alu_ops(info, 1) if prec == gpn.GP_DF64 else {}

    def roof(name, ms):
        return roof_of(ab, name, ms, peak, peak_src, traffic.get(name) if tr_ok else None,
                       alu_ops=alu.get(name))

    result = {
        "metric": METRIC, "value": round(value, 3), "unit": UNIT, "n_gpus": ws, "steps": iters,
        "warmup": args.warmup, "ms_per_step": round(ms_step, 4), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": dtype, "data": "synthetic",
        "config": {"workload": w.name, "N": N, "d": w.d, "nu": w.nu, "eps": w.eps, "R": 1,
                   "precision": args.precision, "arith": arith,
                   "n_t": info["n_t"], "n_sigma": info["n_sigma"], "M": info["M"], "nf": info["nf"],
                   "kernel_width": info["kernel_width"], "tile": info["tile"], "plan_seconds": round(plan_s, 3),
                   "bytes_resident": info["bytes_resident"],
                   "l2": "inputs larger than L2 (fine grids %.2f GB per pass)" % (
                       (info["n_sigma"] + 1) * info["nf"] ** w.d * rs / 1e9),
                   "parallelism": "replicas" if ws > 1 else "single"},
        "roofline": roof(dom_ours, kern_ms[dom_ours]),
        "roofline_phases": [roof(PHASES[q], phase_ms[q]) for q in range(5)],
        "roofline_kernels": [roof(k, ms) for k, ms in kern_ms.items()],
        "dominant_phase": PHASES[dom],
        "phase_ms": {PHASES[q]: round(phase_ms[q], 4) for q in range(5)},
        "phases_recorded": n_rec,
        "timing": dist_stats,
        "clocks": clocks,
        "e2e": e2e,
        "gpu_launches": launches_per_step(own_columns(plan.info)) * iters,
    }
    result.update(extra)
    return result, w, out_sample, plan


def cpu_baseline(w, gpu_out, seconds):
    """The oracle's exact sampled rows of K alpha, timed on this host's cores."""
    from oracle import kernel as okern
    from oracle import rows as orows
    orows.build()
    wp, sig = okern.paper_fields(w.s, w.l, w.d)
    rng = np.random.default_rng(123)
    done, t_used, errs_num, errs_den = 0, 0.0, 0.0, 0.0
    chunk = 64
    while t_used < seconds:
        idx = rng.integers(0, w.N, chunk)
        t0 = time.perf_counter()
        ref = orows.rows(w.points, wp, sig, w.nu, w.alpha, idx)
        t_used += time.perf_counter() - t0
        done += chunk
        if gpu_out is not None:
            errs_num += float(np.sum((gpu_out[idx] - ref) ** 2))
            errs_den += float(np.sum(ref ** 2))
    rows_per_s = done / t_used
    res = {"value": rows_per_s / 1e6, "unit": UNIT, "cores": orows.threads_used(), "kind": "oracle",
           "sample": "%d exact rows of K alpha by direct sum over N=%d (C, OpenMP), %.1f s; full step extrapolated "
                     "as N rows" % (done, w.N, t_used)}
    if gpu_out is not None:
        res["gpu_rel_err_vs_oracle_rows"] = float(np.sqrt(errs_num / errs_den))
    return res


def exact_rows_error(w, got, n_rows, seed):
    """Relative l2 and largest error of `got` on seeded rows against the oracle's exact rows
    of K alpha (direct sums over all N points, float64, host cores)."""
    from oracle import kernel as okern
    from oracle import rows as orows
    orows.build()
    wp, sig = okern.paper_fields(w.s, w.l, w.d)
    idx = np.random.default_rng(seed).choice(w.N, size=n_rows, replace=False)
    ref = orows.rows(w.points, wp, sig, w.nu, w.alpha, idx)
    d = got[idx] - ref
    return {"rel_l2": float(np.linalg.norm(d) / np.linalg.norm(ref)),
            "rel_max": float(np.max(np.abs(d)) / np.max(np.abs(ref)))}


def run_reference(args, ws, rank):
    if rank != 0:
        return
    w = workload(args)
    from oracle import kernel as okern
    from oracle import rows as orows
    orows.build()
    wp, sig = okern.paper_fields(w.s, w.l, w.d)
    rng = np.random.default_rng(7)
    per_step_rows = 128

    def step():
        orows.rows(w.points, wp, sig, w.nu, w.alpha, rng.integers(0, w.N, per_step_rows))

    for _ in range(args.warmup):
        step()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        step()
    dt = (time.perf_counter() - t0) / args.steps
    # one step computes per_step_rows rows; a full CG step needs N rows
    full_step_s = dt * w.N / per_step_rows
    value = w.N / full_step_s / 1e6
    out = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": full_step_s * 1e3, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "config": {"workload": w.name, "N": w.N, "d": w.d, "nu": w.nu, "eps": w.eps, "R": 1},
           "cpu_baseline": {"kind": "oracle", "cores": orows.threads_used(), "value": value, "unit": UNIT,
                            "sample": "each step: %d exact rows of K alpha by direct sum over N=%d; full step "
                                      "extrapolated as N rows" % (per_step_rows, w.N)},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


# ------------------------------------------------------------------ side measurements
def _events_ms(fn, reps):
    import torch
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(reps):
        fn()
    e1.record()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / reps


def measure_config1(dev):
    """d=1, N=2000, Matern 3/2, eps=1e-6 (latency-bound): one matvec and a CG solve to 1e-8, FP64."""
    import torch
    import gpinputs
    import paper_2407_03608_gb300 as gpn
    from paper_2407_03608_gb300 import abi
    w = gpinputs.config_1d()
    plan = gpn.Plan(torch.from_numpy(w.points).to(dev), torch.from_numpy(w.s).to(dev),
                    torch.from_numpy(w.l).to(dev), nu=w.nu, eps=w.eps, precision=gpn.GP_FP64)
    a = torch.from_numpy(w.alpha).to(dev)
    out = torch.empty_like(a)
    for _ in range(5):
        abi.gp_matvec(plan.handle, a, out, 1, 0.0)
    mv_ms = _events_ms(lambda: abi.gp_matvec(plan.handle, a, out, 1, 0.0), 50)
    y = torch.from_numpy(w.y).to(dev)
    x = torch.empty_like(y)
    its = []
    solve_ms = _events_ms(lambda: its.append(abi.gp_cg_solve(plan.handle, y, x, 1, w.eta ** 2, 1e-8, 20000)[1][0]), 3)
    x64 = x.clone()
    # the same solve with FP32 inner CG inside FP64 refinement (residuals on the FP64 plan)
    lo = gpn.Plan(torch.from_numpy(w.points).to(dev), torch.from_numpy(w.s).to(dev), torch.from_numpy(w.l).to(dev),
                  nu=w.nu, eps=w.eps, precision=gpn.GP_FP32, **plan.matched_opts())
    xr = torch.empty_like(y)
    ref_its = []
    ref_ms = _events_ms(lambda: ref_its.append(
        abi.gp_cg_solve_refined(lo.handle, plan.handle, y, xr, 1, w.eta ** 2, 1e-8, 1e-4, 10, 20000)[1][0]), 3)
    ref_err = float((xr - x64).norm() / x64.norm())
    lo.close()
    plan.close()
    return {"workload": w.name, "precision": "fp64", "matvec_us": round(mv_ms * 1e3, 2),
            "cg_solve_ms": round(solve_ms, 3), "cg_iters": int(its[-1]), "rtol": 1e-8,
            "refined_solve": {"precision": "fp32 inner CG, fp64 refinement", "ms": round(ref_ms, 3),
                              "inner_iters": int(ref_its[-1]), "rel_diff_vs_fp64_cg": ref_err}}


def measure_batched(dev, n, block=8, steps=2):
    """The batched workload: the 2-D clustered points, 64 right-hand sides (8 noisy y vectors
    plus 56 +-1 probes), FP32 spread/FFT/step 3/interp with float64 CG reductions.  All 64
    columns share each CG iteration (one gp_cg_solve call, graph-captured blocks of
    iterations); the plan holds grids for `block` columns and runs steps (1)-(5) block after
    block (rhs_block), so 64 columns fit where 64 sets of grids (about 640 GB) would not."""
    import torch
    import gpinputs
    import paper_2407_03608_gb300 as gpn
    from paper_2407_03608_gb300 import abi
    w = gpinputs.config_2d_batched(n)
    R = w.y.shape[1]
    plan = gpn.Plan(torch.from_numpy(w.points).to(dev), torch.from_numpy(w.s).to(dev),
                    torch.from_numpy(w.l).to(dev), nu=1.5, eps=1e-6, precision=gpn.GP_FP32, max_rhs=R,
                    rhs_block=block)
    Y = torch.from_numpy(np.ascontiguousarray(w.y.T)).to(dev)   # (R, N) = column-major N x R
    X = torch.empty_like(Y)
    abi.gp_cg_solve(plan.handle, Y, X, R, w.eta ** 2, 1e-30, 1)
    ms = _events_ms(lambda: abi.gp_cg_solve(plan.handle, Y, X, R, w.eta ** 2, 1e-30, steps), 1) / steps
    nbytes = plan.info["bytes_resident"]
    plan.close()
    return {"workload": w.name, "R": R, "rhs_block": block, "precision": "fp32 (f64 CG)",
            "ms_per_step": round(ms, 3), "value": round(w.N * R / (ms * 1e-3) / 1e6, 3),
            "unit": "Mpts/s (N*R per CG iteration)", "bytes_resident": int(nbytes),
            "columns": "8 noisy y (seeds 10-17) + 56 Rademacher probes (seed 18)"}


def measure_config3(dev, steps=3):
    """d=3, N=2e6 uniform, Matern 5/2, eps=1e-6, FP32: one CG iteration with the stored A'
    tensor and with the memory-lean step 3, and the per-phase milliseconds of each (the
    library's own events)."""
    import torch
    import gpinputs
    import paper_2407_03608_gb300 as gpn
    from paper_2407_03608_gb300 import abi
    w = gpinputs.config_3d()
    pts, s_, l_ = (torch.from_numpy(v).to(dev) for v in (w.points, w.s, w.l))
    y = torch.from_numpy(w.y).to(dev)
    x = torch.empty_like(y)
    out = {"workload": w.name, "precision": "fp32 (f64 CG)", "unit": UNIT}
    opts = None
    for name, s3 in (("stored_a", 1), ("memory_lean_step3", 2)):
        t0 = time.perf_counter()
        plan = gpn.Plan(pts, s_, l_, nu=w.nu, eps=w.eps, precision=gpn.GP_FP32, step3=s3, **(opts or {}))
        torch.cuda.synchronize()
        plan_s = time.perf_counter() - t0
        if opts is None:
            i = plan.info
            opts = dict(plan.matched_opts(), nf=i["nf"])
            out.update(nf=i["nf"], M=i["M"], n_sigma=i["n_sigma"], kernel_width=i["kernel_width"])
        abi.gp_cg_solve(plan.handle, y, x, 1, w.eta ** 2, 1e-30, 1)
        ms = _events_ms(lambda: abi.gp_cg_solve(plan.handle, y, x, 1, w.eta ** 2, 1e-30, steps), 1) / steps
        phase_ms, _, n_rec = _phases(abi, plan, y, x, w.eta ** 2, 2)
        out[name] = {"step3": s3, "ms_per_step": round(ms, 3),
                     "value": round(w.N / (ms * 1e-3) / 1e6, 3), "plan_seconds": round(plan_s, 3),
                     "bytes_resident": int(plan.info["bytes_resident"]),
                     "phase_ms": dict(zip(("spread", "fft_fwd", "step3", "fft_inv", "interp"),
                                          (round(v, 3) for v in phase_ms)))}
        plan.close()
        torch.cuda.empty_cache()
    best = min((v for v in out.values() if isinstance(v, dict)), key=lambda v: v["ms_per_step"])
    out["ms_per_step"], out["value"] = best["ms_per_step"], best["value"]
    return out


def measure_serving(n_requests, n_models=6, max_rhs=4):
    """A bounded sample of the serving stream: requests on `n_models` models (points, fields,
    nu; popularity 1/k), solved to rtol 1e-8 (FP32 CG inside float64 refinement) with each
    model's plans kept resident (PlanCache, 120 GB budget); p50/p99 latency at 80% of the
    measured capacity, one request at a time and with continuous batching (3 slots); every
    10th served solution compared with the plain float64 GPU solve."""
    import gpinputs
    from paper_2407_03608_gb300.serving import Server
    reqs = gpinputs.serving_stream(n_requests, n_min=1000, n_max=20_000, dims=(1, 2), nus=(0.5, 1.5, 2.5),
                                   max_rhs=max_rhs, n_models=n_models)
    srv = Server(hbm_budget=120e9, eps_target=1e-6, cache_plans=True)
    out = srv.serve(reqs, load=0.8, check_every=10)
    out.pop("records")
    # the same stream again with a cold cache and no cache, and with three requests in flight
    srv.cache.clear()
    nocache = Server(hbm_budget=120e9, eps_target=1e-6, cache_plans=False)
    cold = nocache.serve(reqs, load=0.8)
    out["without_cache"] = {k: cold[k] for k in ("capacity_solves_per_s", "latency_p50_s", "latency_p99_s",
                                                 "service_p50_s", "plan_share")}
    out["continuous_batching"] = srv.serve_batched(reqs, load=0.8, slots=3)
    srv.cache.clear()
    out["sample"] = ("%d requests of the serving stream (seed 100) on %d models: N log-uniform in [1e3, 2e4], "
                     "d in {1, 2}, nu in {1/2, 3/2, 5/2}, R in 1..%d (a 2-D model's grid is as large as the "
                     "N = 1e6 workload's, so a request costs seconds per right-hand side; 3-D models cost "
                     "minutes)" % (n_requests, n_models, max_rhs))
    return out


def measure_nu_half(dev, checks, eps=5e-3, near_radius=2e-3):
    """The 2-D clustered workload at nu = 1/2 on the largest grid that fits one GB300 (eps =
    5e-3: nf = 32768, M = 6944; eps = 2.5e-3 would need nf = 65536, 560 GB in FP64): one
    matvec of each of FP64, FP32, both with the exact diagonal correction, and FP64 with the
    diagonal and the near-field correction (pairs closer than near_radius, about ten grid
    wavelengths 1/(M dw)), timed, and their outputs kept for the CPU-baseline leg to compare
    with exact rows of K alpha.
    For nu = 1/2 the mode count grows like eps^-1 (Sec. 5.4), so 1e-6 is out of reach."""
    import torch
    import gpinputs
    import paper_2407_03608_gb300 as gpn
    w = gpinputs.config_2d(1_000_000, 0.5)
    pts, s_, l_ = (torch.from_numpy(v).to(dev) for v in (w.points, w.s, w.l))
    a = torch.from_numpy(w.alpha).to(dev)
    out = {"workload": w.name, "eps": eps}
    opts = None
    for name, prec, dc, r_c in (("fp64", gpn.GP_FP64, 0, 0.0), ("fp64_diag_correct", gpn.GP_FP64, 1, 0.0),
                                ("fp64_diag_near_2e-3", gpn.GP_FP64, 1, near_radius),
                                ("fp32", gpn.GP_FP32, 0, 0.0), ("fp32_diag_correct", gpn.GP_FP32, 1, 0.0)):
        kw = dict(opts or {})
        if dc:
            kw["diag_correct"] = 1
        if r_c > 0:
            kw["near_radius"] = r_c
        t0 = time.perf_counter()
        pl = gpn.Plan(pts, s_, l_, nu=0.5, eps=eps, precision=prec, **kw)
        plan_s = time.perf_counter() - t0
        if opts is None:
            opts = {k: v for k, v in pl.matched_opts().items() if k != "diag_correct"}
            i = pl.info
            out.update(nf=i["nf"], M=i["M"], n_sigma=i["n_sigma"], n_t=i["n_t"], kernel_width=i["kernel_width"],
                       transform=i["transform"])
        pl.matvec(a)
        ms = _events_ms(lambda: pl.matvec(a), 2)
        res = pl.matvec(a).cpu().numpy()
        out[name] = {"ms_per_matvec": round(ms, 3), "bytes_resident": int(pl.info["bytes_resident"]),
                     "plan_seconds": round(plan_s, 2)}
        if r_c > 0:
            out[name]["near_pairs"] = int(pl.info["near_pairs"])
        checks.append(("config2_nu_half." + name, w, res))
        pl.close()
        torch.cuda.empty_cache()
    return out


def side_measurements(args, dev, checks):
    res = {}
    for name, fn in (("config1", lambda: measure_config1(dev)),
                     ("batched", lambda: measure_batched(dev, args.n)),
                     ("config2_nu_half", lambda: measure_nu_half(dev, checks)),
                     ("config3", lambda: measure_config3(dev)),
                     ("served", lambda: measure_serving(args.serve_requests))):
        t0 = time.perf_counter()
        try:
            res[name] = fn()
        except Exception as e:  # recorded, not fatal: the headline line is still printed
            res[name] = {"error": "%s: %s" % (type(e).__name__, str(e)[:200])}
        res[name]["wall_s"] = round(time.perf_counter() - t0, 1)
        print("side %s: %.1f s %s" % (name, res[name]["wall_s"], json.dumps(res[name])), file=sys.stderr, flush=True)
    return res


def run_profile_case(args):
    """One plan and a few matvecs of it, so that an ncu launch filter (-k, -s, -c) sees
    only the plan build and the matvec kernels.  d = 2: the clustered workload (Matern
    3/2); d = 3: uniform in the unit cube (Matern 5/2)."""
    import torch
    import gpinputs
    import paper_2407_03608_gb300 as gpn
    w = gpinputs.config_2d(args.n, 1.5) if args.d == 2 else gpinputs.config_3d(args.n)
    dev = torch.device("cuda", 0)
    prec = getattr(gpn, PRECISIONS[args.precision][0])
    plan = gpn.Plan(torch.from_numpy(w.points).to(dev), torch.from_numpy(w.s).to(dev),
                    torch.from_numpy(w.l).to(dev), nu=w.nu, eps=args.eps, precision=prec,
                    transform=args.transform)
    a = torch.from_numpy(w.alpha).to(dev)
    out = None
    for _ in range(args.matvecs):
        out = plan.matvec(a)
    torch.cuda.synchronize()
    i = plan.info
    print({k: i[k] for k in ("nf", "M", "n_sigma", "kernel_width", "tile", "transform")}, float(out.norm()))
    plan.close()


def run_solve_compare(args):
    """Time to solution on the 2-D workload (N = 1e6, Matern 3/2, eps = 1e-6): plain CG on the
    float64-grade plan (float-float, one right-hand side, no refinement) against the refined
    solve (FP32 inner CG to 1e-4 per refinement step, residuals on the float-float plan),
    both to relative residual --rtol; wall time of each solve (synchronised), iterations, and
    the relative difference of the two solutions.  The native float64 path is timed over 20
    iterations and its time to solution extrapolated to the plain CG's iteration count
    (labelled as such)."""
    import torch
    import paper_2407_03608_gb300 as gpn
    from paper_2407_03608_gb300 import abi
    if args.d == 3:
        return run_solve_3d(args)
    dev = torch.device("cuda", 0)
    w = workload(args)
    pts, s_, l_, y = (torch.from_numpy(v).to(dev) for v in (w.points, w.s, w.l, w.y))
    eta2 = w.eta ** 2
    hi = gpn.Plan(pts, s_, l_, nu=w.nu, eps=w.eps, precision=gpn.GP_DF64)
    lo = gpn.Plan(pts, s_, l_, nu=w.nu, eps=w.eps, precision=gpn.GP_FP32, **hi.matched_opts())
    out = {"workload": w.name, "rtol": args.rtol}

    def timed(fn):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        r = fn()
        torch.cuda.synchronize()
        return r, time.perf_counter() - t0

    (xr, ir), t_ref = timed(lambda: hi.solve_refined(lo, y, eta2, rtol=args.rtol, maxit=200000, outer_max=30))
    out["refined_fp32_inner"] = {"seconds": round(t_ref, 3), "inner_iters": int(ir["iters"][0]),
                                 "relres": float(ir["relres"][0]), "status": int(ir["status"])}
    print(json.dumps(out), file=sys.stderr, flush=True)   # progress: the refined solve alone
    (xp, ip), t_plain = timed(lambda: hi.solve(y, eta2, rtol=args.rtol, maxit=200000))
    out["plain_cg_df64"] = {"seconds": round(t_plain, 3), "iters": int(ip["iters"][0]),
                            "relres": float(ip["relres"][0]), "status": int(ip["status"])}
    d = xr - xp
    out["refined_vs_plain"] = {"rel_l2": float(torch.linalg.norm(d) / torch.linalg.norm(xp)),
                               "rel_max": float(d.abs().max() / xp.abs().max())}
    lo.close()
    p64 = gpn.Plan(pts, s_, l_, nu=w.nu, eps=w.eps, precision=gpn.GP_FP64, **hi.matched_opts())
    x64 = torch.empty_like(y)
    abi.gp_cg_solve(p64.handle, y, x64, 1, eta2, 1e-30, 2)
    ms = _events_ms(lambda: abi.gp_cg_solve(p64.handle, y, x64, 1, eta2, 1e-30, 20), 1) / 20
    out["plain_cg_fp64_extrapolated"] = {"ms_per_iter": round(ms, 3),
                                         "seconds": round(ms * 1e-3 * out["plain_cg_df64"]["iters"], 1),
                                         "note": "20 iterations timed, times the float-float CG's iteration count"}
    p64.close()
    hi.close()
    print(json.dumps(out), flush=True)


def run_solve_3d(args, maxit=400, outer_max=4):
    """The 3-D workload (N = 2e6 uniform, Matern 5/2, eps = 1e-6): the refined solve (FP32
    inner CG, residuals on the float64 plan) to relative residual --rtol, timed.  Both plans
    use the memory-lean step 3, so that they fit one GB300 together (78 + 155 GB); the inner
    iterations of each refinement step are capped at `maxit`, and the steps at `outer_max`,
    to bound the run (status GP_ENOTCONV then, with the float64 residual reached)."""
    import torch
    import gpinputs
    import paper_2407_03608_gb300 as gpn
    dev = torch.device("cuda", 0)
    w = gpinputs.config_3d()
    pts, s_, l_, y = (torch.from_numpy(v).to(dev) for v in (w.points, w.s, w.l, w.y))
    lo = gpn.Plan(pts, s_, l_, nu=w.nu, eps=w.eps, precision=gpn.GP_FP32, step3=2)
    # the FP32 plan's fine grid (nf = 864) for the float64 plan too, with its kernel width
    # chosen for that upsampling: 155 GB instead of 258 GB at its own nf = 1024
    hi = gpn.Plan(pts, s_, l_, nu=w.nu, eps=w.eps, precision=gpn.GP_FP64, step3=2, nf=lo.info["nf"],
                  **lo.matched_opts())
    out = {"workload": w.name, "rtol": args.rtol, "nf": lo.info["nf"], "M": lo.info["M"],
           "bytes_resident": int(lo.info["bytes_resident"] + hi.info["bytes_resident"])}
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    x, info = hi.solve_refined(lo, y, w.eta ** 2, rtol=args.rtol, maxit=maxit, outer_max=outer_max)
    torch.cuda.synchronize()
    out["refined_fp32_inner"] = {"seconds": round(time.perf_counter() - t0, 3), "inner_iters": int(info["iters"][0]),
                                 "relres_fp64": float(info["relres"][0]), "status": int(info["status"])}
    print(json.dumps(out), flush=True)
    lo.close()
    hi.close()


def main():
    args = parse()
    ws, rank, local = dist_setup()
    if args.profile_case:
        run_profile_case(args)
        return
    if args.solve_compare:
        run_solve_compare(args)
        return
    if args.impl == "reference":
        run_reference(args, ws, rank)
        return
    result, w, out_sample, plan = run_ours(args, ws, rank, local)
    plan.close()
    if rank == 0:
        checks = []
        if ws == 1 and args.side:
            import torch
            result["side"] = side_measurements(args, torch.device("cuda", local), checks)
        if ws == 1 and not args.no_cpu_baseline:
            result["cpu_baseline"] = cpu_baseline(w, out_sample, args.cpu_seconds)
            # the oracle's exact rows for the side measurements' outputs (this leg is the one
            # that may run the oracle); each entry lands beside its measurement
            for name, wk, got in checks:
                err = exact_rows_error(wk, got, 1024, seed=31)
                node = result["side"]
                *path, leaf = name.split(".")
                for key in path:
                    node = node.setdefault(key, {})
                node.setdefault(leaf, {})["rel_err_vs_1024_exact_rows"] = err
        print(json.dumps(result), flush=True)
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
