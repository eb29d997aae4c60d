"""Benchmark: eigenpairs/s of the SS / shifted-CG eigensolver on one GB300.

Workload (one "step" = one full eigen-solve through the C ABI: quadrature
setup, shifted CG for every quadrature point and source, moments,
Rayleigh-Ritz, acceptance, eigenpair readback):

  16^3 x 32 lattice (n = 1,572,864), kappa = 0.135, antiperiodic time,
  smooth SU(3) links proj(exp(i 0.5 G)) (seed 4), L = 8 Gaussian sources
  (seed 300), M = 16 moments, tol 1e-12; two line-pair windows (Section 3)
  on the two sides of the spectral gap around zero, [-0.1095, -0.0765] and
  [0.0769, 0.1081], N = 32 points each (64 shifts in one seed recurrence,
  beta = 0.3, N' = 20); each window holds the two lowest eigenvalue
  clusters of its sign, 48 eigenpairs in all.  The sources run one at a
  time (opts.source_block = 1), two such runs side by side on their own
  streams (opts.block_streams = 2), so that the stored seed residuals of the
  two fit the device memory; FP64 throughout ("plain"), the moment
  combination on the tensor cores through an exact fp16 splitting of the
  FP64 operands (as accurate as the FP64 sum; SSQCD_MOMENTS_TC=0 runs it
  on the FP64 pipe).

``value`` counts accepted eigenpairs with residual <= 1e-8 per second of
device time (inputs resident, CUDA events on the library's stream; the
stored residuals, 63 GB a source, are far larger than L2).  ``e2e`` is the
same metric with host inputs (gauge field and sources copied in,
eigenvectors copied out) timed on the host.  Under torchrun every rank
solves an independent replica (its own sources): the path has no data
exchange, so scaling is weak and there is no collective on the data path.

``mixed`` reports the same metric on the same workload for the solve
precision SSQCD_DF (float-float seed vectors, stored
residuals and the Rayleigh-Ritz basis on the FP32 pipes; FP64 recurrence
scalars, eigenvectors and residuals), with
its ratio to the plain FP64 value.  ``mixed_fp32_fp16`` records the FP32
stencil / FP16-link form, which cannot reach the residual bar (it runs on
the 8^4 workload, where it converges).  ``config2`` repeats the plain and
float-float measurements on the 8^4 workload (kappa 0.125, L = 4, N = 32,
M = 8, 12 eigenpairs), whose data fit in L2.  ``serving``,
``serving_16x32`` and ``batched_uneven`` drive the library's request
scheduler: Poisson arrivals on small resident lattices, the headline
lattice resident beside small ones under a memory budget, and 48 uneven
requests over 8^4 / 12^4 / 16^4 lattices submitted at once.

``--impl reference`` times the FP64 numpy oracle on the host cores on a
bounded sample of the same workload (shifted-CG iterations of one source
with all 64 shifts, the moment sums, one Rayleigh-Ritz pass at reduced
width), scaled to a full step by the iteration count of the oracle's own
run of this workload (tests/golden/config3_iterations.json); it also runs
the 4^4 workload of the oracle tests end to end.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "eigenpairs/s at resid<=1e-8 (SS-RR, shifted CG): plain FP64; float-float mixed beside it"
UNIT = "eigenpairs/s"
RES_TOL = 1e-8

WORKLOAD = dict(
    name="16^3x32 smooth eps=0.5 kappa=0.135 L=8 M=16 two windows x N=32 (64 shifts) beta=0.3 FP64",
    dims=(16, 16, 16, 32), kappa=0.135, bc_t=-1, kind="smooth", gauge_seed=4, eps=0.5,
    L=8, src_seed=300, windows=((-0.1095, -0.0765), (0.0769, 0.1081)), N=32, M=16, beta=0.3, nprime=20,
    tol=1e-12, source_block=1, block_streams=2, basis_max_bytes=160e9,
)

CONFIG2 = dict(
    name="8^4 smooth eps=0.3 kappa=0.125 L=4 N=32 M=8 beta=0.6 [0.105,0.120] FP64",
    dims=(8, 8, 8, 8), kappa=0.125, bc_t=-1, kind="smooth", gauge_seed=2, eps=0.3,
    L=4, src_seed=200, N=32, M=8, interval=(0.105, 0.120), beta=0.6, nprime=16, tol=1e-12,
)

# ---- FP64 pipe peak (alu roofline of the FP64 kernels) ---------------------------------
# 152 SMs x 2 FP64 FMA / clock / SM x 2 flop x 2.07 GHz (GB300 FP64 runs at 1/64 of
# FP32); a throughput probe measured 1.19-1.20 TFLOP/s at ~1.98 GHz.
FP64_PEAK_TFLOPS = 152 * 2 * 2 * 2.07e9 / 1e12

# algorithmic cost of one element-shift update of the fused kernel (FP64):
#   y += a p_hat (4 FMA), p_hat = r + b p_hat (4 FMA) -> 16 flop;
#   y, p_hat read and written once -> 64 B.
UPDATE_FLOP_PER_UNIT = 16
UPDATE_BYTES_PER_UNIT = 64
# stencil: 8 hops x (12 projection adds + 6 x 12 link FMA/MUL + 24 reconstruction adds)
# + 24 = 888 FP64 instructions; counted as 1368 flop/site/rhs (FMA = 2); bytes:
# spinor in 192 B + out 192 B + links 576 B (shared by the rhs) per site.
STENCIL_FLOP_PER_SITE = 1368
# The stencil of FP64 lattices in 60-bit fixed point (cg_stencil_kernel<StencilFix<1>>): a
# hop takes 3 products of 32-bit digits for each of the 18 x 4 real products of its two
# link-times-spin-row products; the wide multiply-add runs at 32 lanes a clock and SM.
STENCIL_MADS_PER_SITE = 8 * 2 * 9 * 4 * 3
WIDE_MAD_PEAK = 152 * 32 * 2.07e9 / 1e12
# DRAM traffic of one launch of that kernel (1 rhs, 16^3 x 32) from an ncu capture
# (dram__bytes_read.sum + dram__bytes_write.sum,
# profiles/stencil_integer_fp64_16x16x16x32.md); None once the kernel changes.
STENCIL_FP64_TRAFFIC = 132803584.0 + 12933120.0
# DRAM traffic of one launch of each update kernel with all 128 (source,
# shift) pairs live on this workload (ncu dram__bytes_read.sum +
# dram__bytes_write.sum, one capture per kernel; the algorithmic bytes of such
# a launch are 64 x 128 x 49152 = 402.7 MB -- part of y / p-hat stays in L2).
# Null them when the kernel changes.
# DRAM traffic of one launch of basis_combine_kernel on the headline workload
# (one window, one block of 2 sources, 2499 stored residuals, 16 moments,
# real coefficients) from a one-pass ncu capture (dram__bytes_read.sum
# 123.875 GB + dram__bytes_write.sum 0.814 GB); None once the kernel changes.
COMBINE_TRAFFIC = 123875257344.0 + 814184960.0
UPDATE_FP64_TRAFFIC_ALL_LIVE = (204.503552 + 139.793408) * 1e6
UPDATE_TMA_TRAFFIC_ALL_LIVE = (204.504320 + 139.588352) * 1e6


def _measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        return json.load(open(p))
    return {"hbm_gbs": 6800.0, "fallback": True}


class ClockSampler:
    """nvidia-smi SM clocks and throttle reasons during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None

    def start(self):
        import tempfile
        try:
            fd, self.path = tempfile.mkstemp(prefix="ssqcd_clocks_", suffix=".csv")
            self.f = os.fdopen(fd, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.f.close()
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax = float(parts[2])
            except ValueError:
                continue
            for nm, val in zip(names, parts[5:9]):
                if val.lower() == "active":
                    reasons.add(nm)
        try:
            os.unlink(self.path)
        except OSError:
            pass
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm)}


def _dist():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def reduce_job(ms, pairs, world, device):
    """Whole-job numbers of independent replicas: the slowest rank's time
    and the eigenpairs of all ranks (no data-path collective; this is the
    only exchange)."""
    if world <= 1:
        return ms, pairs
    import torch
    import torch.distributed as dist
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    c = torch.tensor([pairs], dtype=torch.float64, device=device)
    dist.all_reduce(c, op=dist.ReduceOp.SUM)
    return float(t.item()), float(c.item())


def make_inputs(rank=0, w=None):
    import synthetic
    w = WORKLOAD if w is None else w
    U = synthetic.gauge_field(w["dims"], w["kind"], seed=w["gauge_seed"], eps=w["eps"])
    src = synthetic.gaussian_sources(w["dims"], w["L"], seed=w["src_seed"] + 1000 * rank)
    return U, src


def windows_step(ss, lat, src, w, want_vectors=False):
    """One solve of the headline workload: (evals, residuals, stats[, evecs])."""
    res = ss.ss_solve_windows(lat, w["windows"], w["N"], w["M"], src, beta=w["beta"], nprime=w["nprime"],
                              tol=w["tol"], source_block=w["source_block"], basis_max_bytes=w["basis_max_bytes"],
                              block_streams=w.get("block_streams", 1))
    if res.status != ss.OK:
        raise RuntimeError(f"solve failed with status {res.status}: {res.error}")
    ev, vec, rs, st = ss.ss_eigpairs(res, want_vectors=want_vectors)
    return (ev, rs, st, vec) if want_vectors else (ev, rs, st)


def moments_flops(w, st, n):
    """Algorithmic FP64 flops of the moment combination of one solve:
    (windows x M) moments x (slots = iterations + 1) stored residuals x n
    complex elements x L sources (each block's slot count is bounded by the
    largest, stats.iterations), times 4 per term when the coefficients are
    real (stats.real_moments: a real times a complex number, 2 FMA) and 8
    when they are complex (a complex multiply-add)."""
    per = 4 if st.get("real_moments") else 8
    return per * len(w["windows"]) * w["M"] * (st["iterations"] + 1) * n * w["L"]


def moments_roofline(w, st, n, mom_tf, step_ms, peaks):
    """Roofline line of the moment combination.  With real coefficients and
    FP64 residuals it runs on the tensor cores (combine_tc_kernel, unless
    SSQCD_MOMENTS_TC=0): exact fp16 slices, so its roof is reading the
    stored residuals once (16 B a complex element and slot, each window);
    the phase also holds the scale pass, which reads them once more a
    window.  Otherwise the FP64-pipe kernel, bound by the FP64 rate."""
    tc = bool(st.get("real_moments")) and os.environ.get("SSQCD_MOMENTS_TC", "1") != "0"
    if tc:
        nbytes = 16.0 * len(w["windows"]) * (st["iterations"] + 1) * n * w["L"]
        gbs = nbytes / (st["ms_moments"] / 1e3) / 1e9
        return {
            "kernel": "combine_tc_kernel (moments on the tensor cores: the FP64 residuals and real coefficients "
                      "cut exactly into seven 8-bit fp16 slices, 28 slice-pair tcgen05.mma into tensor memory, "
                      "exact integer sums; with its scale pass, one read of the residuals more)",
            "bound": "hbm", "achieved": gbs, "peak": peaks["hbm_gbs"], "unit": "GB/s",
            "frac": gbs / peaks["hbm_gbs"], "traffic": None,
            "traffic_note": "no ncu capture of this kernel; algorithmic bytes: each stored residual read once "
                            "a window (windows x slots x n x 16 B a source)",
            "fp64_equivalent_tflops": mom_tf,
            "fp64_equivalent_note": "4 flop a term (real coefficient times complex element) over the phase time, "
                                    "against the FP64 pipe's 1.259 TFLOP/s",
            "phase_ms": st["ms_moments"], "fraction_of_step": st["ms_moments"] / step_ms,
        }
    return {
        "kernel": "basis_combine_kernel (moments from the stored seed residuals, FP64; the moments phase, "
                  "whose other kernels are the small coefficient recurrences)",
        "bound": "alu", "achieved": mom_tf, "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s",
        "frac": mom_tf / FP64_PEAK_TFLOPS, "traffic": COMBINE_TRAFFIC,
        "traffic_note": "bytes per launch (one window, one block of 2 sources: each residual read "
                        "once, 2 x 2499 x 1572864 x 16 B = 125.8 GB, and 32 moments written, 0.8 GB; "
                        "profiles/combine_fp64_16x16x16x32.md); the headline runs one source a launch",
        "flop_count": ("4 per term: real coefficients (conjugate-pair points), a real times a complex "
                       "residual element, 2 FMA" if st.get("real_moments") else
                       "8 per complex multiply-add (the kernel issues 3 real multiplications per product)"),
        "phase_ms": st["ms_moments"], "fraction_of_step": st["ms_moments"] / step_ms,
    }


def run_ours(args):
    import torch
    import torch.distributed as dist

    import paper_1004_0292_gb300 as ss
    from paper_1004_0292_gb300 import build as ssbuild

    world, rank, local = _dist()
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    ssbuild.build()
    w = WORKLOAD
    U, src = make_inputs(rank)
    # a side stream: the legacy default stream cannot be captured into the
    # library's CUDA graphs
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    lat = ss.create_lattice(w["dims"], w["kappa"], w["bc_t"], stream=stream)
    U_d = torch.from_numpy(U).cuda()
    src_d = torch.from_numpy(src).cuda()
    ss.upload_gauge(lat, U_d)
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")  # 256 MB > L2
    n = 12 * int(np.prod(w["dims"]))
    V = int(np.prod(w["dims"]))
    peaks = _measured_peaks()

    def step():
        return windows_step(ss, lat, src_d, w)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clocks = ClockSampler(local)
    clocks.start()
    launches0 = ss.kernel_launches()
    times, counts, plain, res_p = timed_steps(step, flush, stream, args.steps)
    torch.cuda.synchronize()
    launches = ss.kernel_launches() - launches0
    clk = clocks.stop()
    total_ms, total_pairs = reduce_job(float(sum(times)), float(sum(counts)), world, "cuda")
    value = total_pairs / (total_ms / 1e3)
    # per-kernel device times: a separate step with the library's sampled
    # kernel timing on (its event nodes slow the loop a little, so they stay
    # out of the timed steps above)
    # (one run at a time there, so that each kernel's events see only its own run)
    w_kt = dict(w, block_streams=1)
    ss.set_kernel_timing(True)
    _, _, stats, _ = timed_steps(lambda: windows_step(ss, lat, src_d, w_kt), flush, stream, KERNEL_TIMING_STEPS)
    ss.set_kernel_timing(False)

    # ---- rooflines: the moment combination and the stencil ----
    last = plain[-1]
    mflops = moments_flops(w, last, n)
    mom_tf = mflops / (last["ms_moments"] / 1e3) / 1e12
    # the stencil of the CG loop (second kernel): events on one chunk in four
    it_tot = sum(s["launches_update"] for s in stats)
    ms_sten = sum(s["ms_k_stencil"] for s in stats)
    Lb = w["source_block"]
    # shifted-CG runs one after another: groups of block_streams runs of Lb sources side by side
    n_groups = -(-w["L"] // (Lb * w.get("block_streams", 1)))
    sten_flops = it_tot * V * Lb * STENCIL_FLOP_PER_SITE
    sten_bytes = it_tot * V * (Lb * 3 * 192 + 576)  # p and its digits in, q out, the links' digits
    sten_tf = sten_flops / (ms_sten / 1e3) / 1e12 if ms_sten > 0 else None
    sten_mads = it_tot * V * Lb * STENCIL_MADS_PER_SITE / (ms_sten / 1e3) / 1e12 if ms_sten > 0 else None

    # ---- end to end through the C ABI with host buffers ----
    e2e = None
    if not args.no_e2e:
        e2e_times, e2e_pairs = [], []
        h2d = U.nbytes + src.nbytes
        d2h = 0
        for _ in range(max(1, min(args.e2e_steps, args.steps))):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            lat2 = ss.create_lattice(w["dims"], w["kappa"], w["bc_t"], stream=stream)
            ss.upload_gauge(lat2, U)
            ev, rs, st, vec = windows_step(ss, lat2, src, w, want_vectors=True)
            torch.cuda.synchronize()
            e2e_times.append(time.perf_counter() - t0)
            e2e_pairs.append(int(np.sum(rs <= RES_TOL)))
            d2h = ev.nbytes + rs.nbytes + vec.nbytes
            del lat2, vec
        e2e = {"value": float(sum(e2e_pairs) / sum(e2e_times)), "unit": UNIT,
               "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h)}

    # ---- mixed arm: float-float seed vectors and stored residuals (SSQCD_DF) ----
    mixed = None
    if not args.no_mixed:
        lat_m = ss.create_lattice(w["dims"], w["kappa"], w["bc_t"], precision=ss.DF, stream=stream)
        ss.upload_gauge(lat_m, U_d)

        def step_m():
            return windows_step(ss, lat_m, src_d, w)

        for _ in range(args.warmup):
            step_m()
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()
        t_m, c_m, p_m, res_m = timed_steps(step_m, flush, stream, args.steps)
        r_m = [float(np.max(rs[rs <= RES_TOL])) if np.any(rs <= RES_TOL) else None for rs in res_m]
        ss.set_kernel_timing(True)
        _, _, s_m, _ = timed_steps(lambda: windows_step(ss, lat_m, src_d, dict(w, block_streams=1)), flush, stream,
                                   KERNEL_TIMING_STEPS)
        ss.set_kernel_timing(False)
        ms_m, pairs_m = reduce_job(float(sum(t_m)), float(sum(c_m)), world, "cuda")
        value_m = pairs_m / (ms_m / 1e3)
        it_m = max(1, sum(x["launches_update"] for x in s_m))
        mixed = {
            "precision": "SSQCD_DF: float-float (FP32 pair, 48-bit significand) seed vectors and stored residuals, and "
                         "the Rayleigh-Ritz basis and products, on the FP32 pipes; links and hops in 60-bit fixed point; "
                         "FP64 recurrence scalars, eigenvectors and residuals",
            "value": value_m, "unit": UNIT, "ms_per_step": ms_m / args.steps,
            "vs_plain_fp64": value_m / value, "eigenpairs_per_step": c_m[-1],
            "max_accepted_residual": r_m[-1], "iterations_per_step": p_m[-1]["iterations"],
            "phase_ms": {"cg": p_m[-1]["ms_cg"], "moments": p_m[-1]["ms_moments"], "rr": p_m[-1]["ms_rr"]},
            "cg_us_per_iteration": 1e3 * p_m[-1]["ms_cg"] / max(1, p_m[-1]["iterations"]) / n_groups,
            "kernel_us_per_iteration": {"stencil": 1e3 * sum(x["ms_k_stencil"] for x in s_m) / it_m,
                                        "seed_update": 1e3 * sum(x["ms_k_seed"] for x in s_m) / it_m,
                                        "seed_direction": 1e3 * sum(x["ms_k_scalars"] for x in s_m) / it_m,
                                        "timed_iterations": it_m},
        }
        # the float-float arm's dominant kernel: its stencil (one rhs a launch)
        sten_us_m = 1e3 * sum(x["ms_k_stencil"] for x in s_m) / it_m
        sten_gbs_m = V * (Lb * 3 * 192 + 576) / (sten_us_m * 1e-6) / 1e9 if sten_us_m > 0 else None
        mixed["stencil"] = {
            "kernel": "cg_stencil_kernel<StencilFix<1, float4>> (q = K p with the (p, q) partials: hops in 60-bit "
                      "fixed point, the rest in float-float)",
            "bound": "integer multiply-adds and their latency at 16 warps an SM",
            "avg_launch_us": sten_us_m, "rhs_per_launch": Lb, "hbm_achieved_gbs": sten_gbs_m,
            "hbm_frac": sten_gbs_m / peaks["hbm_gbs"] if sten_gbs_m else None,
            "note": "algorithmic bytes 192 + 192 in (p and its digits) + 192 out + 576 links a site",
            "share_of_step": (sten_us_m * p_m[-1]["iterations"] * w["L"] / Lb) / 1e3 / (ms_m / args.steps),
        }
        del lat_m

    config2 = None
    if not args.no_config2:
        config2 = run_config2(ss, stream, flush, args, world, peaks)

    stencil_large = None
    if not args.no_serving:
        stencil_large = run_stencil_large(ss, stream, peaks)

    serving = serving_large = batched = None
    if not args.no_serving:
        U8, _ = make_inputs(rank, CONFIG2)
        serving = run_serving(ss, stream, U8, seed=17 + rank)
        serving_large = run_serving_large(ss, stream, U, src, U8, seed=23 + rank)
        batched = run_batched_uneven(ss, stream)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(budget_s=args.cpu_budget, gpu_iterations=last["iterations"], pairs=counts[-1])

    if rank == 0:
        lat_sorted = sorted(times)
        r_p = [float(np.max(rs[rs <= RES_TOL])) if np.any(rs <= RES_TOL) else None for rs in res_p]
        out = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic (seeded smooth SU(3) links, Gaussian sources)",
            "config": {"workload": w["name"], "lattice": list(w["dims"]), "kappa": w["kappa"],
                       "sources": w["L"], "source_block": w["source_block"],
                       "block_streams": w.get("block_streams", 1), "windows": [list(x) for x in w["windows"]],
                       "quad_points_per_window": w["N"], "shifts": w["N"] * len(w["windows"]), "moments": w["M"],
                       "beta": w["beta"], "nprime": w["nprime"], "tol": w["tol"],
                       "parallelism": f"replicas x{world}",
                       "l2": "inputs larger than L2 (stored residuals 63 GB per source, two sources resident) and a 256 MB "
                             "flush write between steps"},
            "eigenpairs_per_step": counts[-1], "max_accepted_residual": r_p[-1],
            "iterations_per_step": last["iterations"],
            "latency_ms": {"p50": float(np.percentile(lat_sorted, 50)), "p99": float(np.percentile(lat_sorted, 99))},
            "phase_ms": {"cg": last["ms_cg"], "moments": last["ms_moments"], "rr": last["ms_rr"]},
            "cg_us_per_iteration": 1e3 * last["ms_cg"] / max(1, last["iterations"]) / n_groups,
            "stored_residual_bytes_per_block": last["basis_bytes"],
            "roofline": {
                "kernel": "cg_stencil_kernel<StencilFix<1>> (q = K p with the (p, q) partials: hops in 60-bit fixed "
                          "point on the integer multiply-adds; the step's dominant kernel: 2 x L x iterations launches)",
                "bound": "alu", "achieved": sten_mads, "peak": WIDE_MAD_PEAK,
                "unit": "T 32 x 32 + 64-bit integer multiply-adds/s",
                "frac": sten_mads / WIDE_MAD_PEAK if sten_mads else None, "traffic": STENCIL_FP64_TRAFFIC,
                "traffic_note": "one launch; algorithmic 192 + 192 B of digits and p in, 192 out, 576 of links a site = "
                                "151 MB",
                "peak_source": "derived: 152 SMs x 32 lanes/clk (measured by a probe) x 2.07 GHz (no integer entry in "
                               "MEASURED_PEAKS.json)",
                "op_count": "1728 a site and rhs: 8 hops x 18 complex products x 4 real ones x 3 digit products",
                "fp64_equivalent_tflops": sten_tf,
                "fp64_equivalent_note": "1368 flop a site and rhs (the Wilson hop's 1320 plus gamma5 and the diagonal; "
                                        "FMA = 2), beside the FP64 pipe's 1.259 TFLOP/s",
                "avg_launch_us": 1e3 * ms_sten / max(1, it_tot), "rhs_per_launch": Lb,
                "hbm_achieved_gbs": sten_bytes / (ms_sten / 1e3) / 1e9 if ms_sten > 0 else None,
                "launch_time_source": "a separate step with the library's kernel timing on (one run at a time): "
                                      "CUDA events on the launching stream, one 16-iteration chunk in four",
                "share_of_step": (ms_sten / max(1, it_tot) * last["iterations"] * w["L"] / Lb)
                                 / (total_ms / args.steps),
            },
            "moments_roofline": moments_roofline(w, last, n, mom_tf, total_ms / args.steps, peaks),
            "kernel_us_per_iteration": {"stencil": 1e3 * ms_sten / max(1, it_tot),
                                        "seed_update": 1e3 * sum(s["ms_k_seed"] for s in stats) / max(1, it_tot),
                                        "seed_direction": 1e3 * sum(s["ms_k_scalars"] for s in stats) / max(1, it_tot),
                                        "timed_iterations": it_tot, "rhs": Lb},
            "e2e": e2e, "cpu_baseline": cpu, "clocks": clk, "gpu_launches": int(launches), "mixed": mixed,
            "mixed_fp32_fp16": config2.pop("fp32_fp16") if config2 else None,
            "config2": config2, "serving": serving, "serving_16x32": serving_large, "batched_uneven": batched,
            "stencil_large": stencil_large,
        }
        print(json.dumps(out), flush=True)
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()


def run_config2(ss, stream, flush, args, world, peaks):
    """The 8^4 workload (data in L2): plain FP64 and float-float eigenpairs/s,
    the FP64 stencil's roofline there, the update form, and the FP32 / FP16
    link path's residuals."""
    import torch
    w = CONFIG2
    U, src = make_inputs(0, w)
    U_d = torch.from_numpy(U).cuda()
    src_d = torch.from_numpy(src).cuda()
    n = 12 * int(np.prod(w["dims"]))
    V = int(np.prod(w["dims"]))
    out = {"workload": w["name"]}
    steps = max(3, args.steps)
    for name, prec in (("plain_fp64", ss.FP64), ("float_float", ss.DF), ("fp32_fp16", ss.MIXED)):
        lat = ss.create_lattice(w["dims"], w["kappa"], w["bc_t"], precision=prec, stream=stream)
        ss.upload_gauge(lat, U_d)

        def step(basis=1, lat=lat):
            res = ss.ss_solve(lat, w["interval"], w["N"], w["M"], src_d, beta=w["beta"], nprime=w["nprime"],
                              tol=w["tol"], basis=basis)
            if res.status != ss.OK:
                raise RuntimeError(f"solve failed with status {res.status}: {res.error}")
            ev, _, rs, st = ss.ss_eigpairs(res, want_vectors=False)
            return ev, rs, st

        for _ in range(args.warmup):
            step()
        times, counts, plain, res = timed_steps(step, flush, stream, steps)
        ms, pairs = reduce_job(float(sum(times)), float(sum(counts)), world, "cuda")
        ent = {"value": pairs / (ms / 1e3), "unit": UNIT, "ms_per_step": ms / steps,
               "eigenpairs_per_step": counts[-1], "accepted_per_step": int(len(res[-1])),
               "max_accepted_residual": float(np.max(res[-1])) if len(res[-1]) else None,
               "iterations_per_step": plain[-1]["iterations"],
               "cg_us_per_iteration": 1e3 * plain[-1]["ms_cg"] / max(1, plain[-1]["iterations"])}
        if name == "fp32_fp16":
            ent["precision"] = ("SSQCD_MIXED: FP32 stencil and shift vectors with FP16 12-parameter links; no "
                                "accepted pair reaches residual 1e-8 (the FP16 links perturb A by ~5e-4), and on "
                                "the 16^3 x 32 workload the FP32 seed recurrence does not converge")
        if name == "plain_fp64":
            ss.set_kernel_timing(True)
            _, _, stats, _ = timed_steps(step, flush, stream, KERNEL_TIMING_STEPS)
            ss.set_kernel_timing(False)
            it_tot = sum(s["launches_update"] for s in stats)
            ms_sten = sum(s["ms_k_stencil"] for s in stats)
            tf = it_tot * V * w["L"] * STENCIL_FLOP_PER_SITE / (ms_sten / 1e3) / 1e12
            mads = tf / STENCIL_FLOP_PER_SITE * STENCIL_MADS_PER_SITE
            ent["stencil"] = {"kernel": "cg_stencil_kernel<StencilFix<1>>", "bound": "alu", "achieved": mads,
                              "unit": "T 32 x 32 + 64-bit integer multiply-adds/s", "frac": mads / WIDE_MAD_PEAK,
                              "fp64_equivalent_tflops": tf, "traffic": None,
                              "avg_launch_us": 1e3 * ms_sten / max(1, it_tot)}
            ent["kernel_us_per_iteration"] = {
                "stencil": 1e3 * ms_sten / max(1, it_tot),
                "seed_update": 1e3 * sum(s["ms_k_seed"] for s in stats) / max(1, it_tot),
                "seed_direction": 1e3 * sum(s["ms_k_scalars"] for s in stats) / max(1, it_tot)}
            if not args.no_update_form:
                ent["update_form"] = run_update_form(step, stream, flush, args, n, world)
        out[name] = ent
        del lat
    out["float_float_vs_plain"] = out["float_float"]["value"] / out["plain_fp64"]["value"]
    return out


KERNEL_TIMING_STEPS = 1


def timed_steps(step, flush, stream, k, **kw):
    """k solves, each timed with CUDA events on the library's stream after an
    L2 flush: (ms list, accepted-pair counts, stats list, residual arrays)."""
    import torch
    times, counts, stats, res = [], [], [], []
    for _ in range(k):
        flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record(stream)
        ev, rs, st = step(**kw)
        e1.record(stream)
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
        counts.append(int(np.sum(rs <= RES_TOL)))
        stats.append(st)
        res.append(rs)
    torch.cuda.synchronize()
    return times, counts, stats, res


def run_update_form(step, stream, flush, args, n, world):
    """The same FP64 solve with the per-iteration shift-vector updates
    (opts.basis = 0): value, loop time and the update kernel's FP64 roofline."""
    import paper_1004_0292_gb300 as ss
    for _ in range(args.warmup):
        step(basis=0)
    times, counts, plain, _ = timed_steps(step, flush, stream, args.steps, basis=0)
    ms, pairs = reduce_job(float(sum(times)), float(sum(counts)), world, "cuda")
    ss.set_kernel_timing(True)
    _, _, stats, _ = timed_steps(step, flush, stream, KERNEL_TIMING_STEPS, basis=0)
    ss.set_kernel_timing(False)
    ms_upd = sum(s["ms_k_update"] for s in stats)
    units = sum(s["timed_shift_updates"] for s in stats) * n
    it = max(1, sum(s["launches_update"] for s in stats))
    tf = UPDATE_FLOP_PER_UNIT * units / (ms_upd / 1e3) / 1e12 if ms_upd > 0 else None
    return {"value": pairs / (ms / 1e3), "unit": UNIT, "ms_per_step": ms / args.steps, "basis": plain[-1]["basis"],
            "phase_ms": {"cg": plain[-1]["ms_cg"], "moments": plain[-1]["ms_moments"], "rr": plain[-1]["ms_rr"]},
            "cg_us_per_iteration": 1e3 * plain[-1]["ms_cg"] / max(1, plain[-1]["iterations"]),
            "update_kernel": {"kernel": "cg_update_pf_kernel (fused multi-shift update, FP64)",
                              "achieved_tflops": tf, "frac_fp64_peak": tf / FP64_PEAK_TFLOPS if tf else None,
                              "avg_launch_us": 1e3 * ms_upd / it, "traffic": UPDATE_FP64_TRAFFIC_ALL_LIVE,
                              "traffic_note": "one launch with all 128 shift vectors live; algorithmic 402.7 MB"}}


STENCIL_LARGE = dict(dims=(16, 16, 16, 32), kappa=0.135, eps=0.5, gauge_seed=4, rhs=8, reps=20)


def run_stencil_large(ss, stream, peaks, rhs=None):
    """The stencil alone on the mixed-path lattice shape (16^3 x 32, 8
    right-hand sides unless ``rhs`` says otherwise, smooth links eps 0.5,
    kappa 0.135) where its data no longer fits in L2: FP64, float-float and
    FP32 spinors with FP16 / FP32 12-parameter links.  Algorithmic bytes per
    application: spinors in and out for every rhs plus the links once
    (shared by the rhs)."""
    import synthetic
    c = dict(STENCIL_LARGE) if rhs is None else dict(STENCIL_LARGE, rhs=int(rhs))
    U = synthetic.gauge_field(c["dims"], "smooth", seed=c["gauge_seed"], eps=c["eps"])
    V = int(np.prod(c["dims"]))
    out = {"lattice": "x".join(map(str, c["dims"])), "rhs": c["rhs"],
           "note": "device time of the stencil kernel alone, CUDA events, mean of 20 applications"}
    for name, prec, cplx, link_b in (("fp64", ss.FP64, 16, 576), ("float_float", ss.DF, 16, 576),
                                     ("fp32_fp16links", ss.MIXED, 8, 96), ("fp32_fp32links", ss.MIXED_F32LINKS, 8, 192)):
        lat = ss.create_lattice(c["dims"], c["kappa"], -1, precision=prec, stream=stream)
        ss.upload_gauge(lat, U)
        ms = ss.time_stencil(lat, c["rhs"], c["reps"])
        byts = c["rhs"] * V * 2 * 12 * cplx + V * link_b
        gbs = byts / (ms / 1e3) / 1e9
        out[name] = {"us_per_call": 1e3 * ms, "hbm_gbs": gbs, "hbm_frac": gbs / peaks["hbm_gbs"],
                     "tflops": STENCIL_FLOP_PER_SITE * V * c["rhs"] / (ms / 1e3) / 1e12}
        if prec in (ss.MIXED, ss.MIXED_F32LINKS):
            try:
                v, us = ss.stencil_tuning(lat, c["rhs"])
            except ss.SsqcdError:  # a forced variant: nothing tuned
                v, us = None, None
            out[name]["variant"] = {"chosen": v, "us_per_variant": us,
                                    "variants": ["all rhs of 32 sites a block, 4 blocks/SM", "same, 3 blocks/SM",
                                                 "thread per site and rhs pair, 4 blocks/SM", "same, 3 blocks/SM",
                                                 "thread per site and rhs pair, the two rhs in the paired lanes, "
                                                 "4 blocks/SM", "same, 3 blocks/SM",
                                                 "the same with the x-y plane and its y-halo staged in shared "
                                                 "memory, 4 blocks/SM", "same, 3 blocks/SM"]}
        del lat
    return out


SERVING = dict(n_requests=24, rate_per_s=20.0, lattices=("8^4 bench field", "4^4 Haar kappa 0.13"),
               sources=(1, 2, 3, 4), points=(16, 32))


def run_serving(ss, stream, U8, seed=17):
    """Poisson-arrival eigen-window requests on two resident lattices (the
    8^4 bench field and a 4^4 Haar field, kappa 0.13), driven through the
    library's request scheduler; once with plain FP64 lattices and once with
    float-float ones (SSQCD_DF).  Each request: its
    lattice's known interval, L in {1..4} Gaussian sources, N in {16, 32}
    points.  Two arrival patterns of the same requests: exponential gaps
    with mean 1/20 s (seeded; latency under load) and all at once (the GPU
    saturated; throughput).  Reports p50/p99 latency (submission to result)
    and eigenpairs/s at residual <= 1e-8 over the span from the first arrival
    to the last completion."""
    import synthetic
    w = CONFIG2
    dims4 = (4, 4, 4, 4)
    U4 = synthetic.gauge_field(dims4, "haar", seed=1)
    rng = np.random.default_rng(seed)
    cfg = SERVING
    arrivals = np.cumsum(rng.exponential(1.0 / cfg["rate_per_s"], cfg["n_requests"]))
    plan = []
    for i in range(cfg["n_requests"]):
        big = bool(rng.random() < 0.5)
        L = int(rng.choice(cfg["sources"]))
        N = int(rng.choice(cfg["points"]))
        if big:
            src = synthetic.gaussian_sources(w["dims"], L, seed=5000 + i)
            plan.append(("8", w["interval"], N, w["M"], src, dict(beta=w["beta"], nprime=min(w["nprime"], N))))
        else:
            src = synthetic.gaussian_sources(dims4, L, seed=6000 + i)
            plan.append(("4", (0.374, 0.3930), N, 8, src, dict(beta=0.3, nprime=min(14, N))))
    out = {"requests": cfg["n_requests"], "arrivals": f"Poisson, mean {cfg['rate_per_s']}/s, seed {seed}",
           "mix": "half 8^4 (bench field, its 12-eigenpair window), half 4^4 Haar (8-eigenpair window); "
                  "L in 1..4, N in {16, 32}"}
    def serve(lats, arrive):
        srv = ss.Server()
        ids = []
        t0 = time.perf_counter()
        nxt = 0
        while True:
            now = time.perf_counter() - t0
            while nxt < len(plan) and arrive[nxt] <= now:
                key, iv, N, M, src, kw = plan[nxt]
                ids.append(srv.submit(lats[key], iv, N, M, src, **kw))
                nxt += 1
            q, r, f = srv.counts()
            if nxt == len(plan) and q == 0 and r == 0:
                break
            if r > 0 or q > 0:
                srv.progress(wait=(nxt == len(plan) or arrive[nxt] - now > 0.002))
            else:
                time.sleep(max(0.0, arrive[nxt] - now))
        t_end = time.perf_counter() - t0
        lat_ms, pairs, failed = [], 0, 0
        for i in ids:
            state, ms = srv.status(i)
            lat_ms.append(ms)
            res = srv.take(i)
            if res.status != ss.OK:
                failed += 1
                continue
            _, _, rs, _ = ss.ss_eigpairs(res, want_vectors=False)
            pairs += int(np.sum(rs <= RES_TOL))
        deferred = srv.deferred()
        srv.close()
        return {"eigenpairs_per_s": pairs / (t_end - arrive[0]), "eigenpairs": pairs, "failed": failed,
                "waited_on_memory": deferred,
                "latency_ms": {"p50": float(np.percentile(lat_ms, 50)), "p99": float(np.percentile(lat_ms, 99))},
                "span_s": t_end - arrive[0]}

    for name, prec in (("plain_fp64", ss.FP64), ("mixed", ss.DF)):
        lats = {"8": ss.create_lattice(w["dims"], w["kappa"], w["bc_t"], precision=prec, stream=stream),
                "4": ss.create_lattice(dims4, 0.13, -1, precision=prec, stream=stream)}
        ss.upload_gauge(lats["8"], U8)
        ss.upload_gauge(lats["4"], U4)
        out[name] = {"poisson": serve(lats, arrivals),
                     "burst": serve(lats, np.zeros(len(plan)))}
    out["burst_mixed_vs_plain"] = (out["mixed"]["burst"]["eigenpairs_per_s"]
                                   / out["plain_fp64"]["burst"]["eigenpairs_per_s"])
    return out


def _oracle_iterations():
    """Seed iterations of the oracle's own shifted-CG run of the headline
    workload (source 0), from tests/golden/config3_iterations.json (written
    by tests/golden/make_config3_iterations.py), or None when absent or for
    other parameters."""
    path = os.path.join(ROOT, "tests", "golden", "config3_iterations.json")
    if not os.path.exists(path):
        return None
    g = json.load(open(path))
    p, w = g["params"], WORKLOAD
    same = (tuple(p["dims"]) == tuple(w["dims"]) and p["kappa"] == w["kappa"] and p["eps"] == w["eps"]
            and p["gauge_seed"] == w["gauge_seed"] and p["N"] == w["N"] and p["nprime"] == w["nprime"]
            and p["beta"] == w["beta"] and [list(x) for x in p["windows"]] == [list(x) for x in w["windows"]]
            and p["src_seed"] == w["src_seed"] and p["tol"] == w["tol"])
    return int(g["seed_iterations"]) if same else None


def _host_cores():
    try:
        import threadpoolctl
        info = threadpoolctl.threadpool_info()
        return max([i.get("num_threads", 1) for i in info] + [1])
    except Exception:
        return os.cpu_count() or 1


SERVING_LARGE = dict(rate_per_s=20.0, budget_bytes=220e9, n_small=6)


def run_serving_large(ss, stream, U3, src3, U8, seed=23):
    """The scheduler with the headline lattice resident: requests on the
    16^3 x 32 field (the headline's two windows, and its positive window
    alone; L = 8 in source blocks of two, 128 GB of stored residuals a block)
    mixed with small 8^4 and 4^4 requests, Poisson arrivals (mean 20/s,
    seeded), and a 220 GB memory budget, so that the large requests cannot
    run together and admission defers them.  Plain FP64 and float-float
    lattices.  Reports p50/p99 latency, eigenpairs/s at residual <= 1e-8 over
    the span, and how many requests waited on memory."""
    import torch

    import synthetic
    w, w8 = WORKLOAD, CONFIG2
    dims4 = (4, 4, 4, 4)
    U4 = synthetic.gauge_field(dims4, "haar", seed=1)
    rng = np.random.default_rng(seed)
    plan = [("16", [list(x) for x in w["windows"]], src3), ("16", [list(w["windows"][1])], src3)]
    for i in range(SERVING_LARGE["n_small"]):
        if i % 2 == 0:
            plan.append(("8", [list(w8["interval"])], synthetic.gaussian_sources(w8["dims"], 4, seed=7000 + i)))
        else:
            plan.append(("4", [[0.374, 0.3930]], synthetic.gaussian_sources(dims4, 3, seed=7100 + i)))
    order = rng.permutation(len(plan))
    plan = [plan[i] for i in order]
    arrive = np.cumsum(rng.exponential(1.0 / SERVING_LARGE["rate_per_s"], len(plan)))
    kw = {"16": dict(N=w["N"], M=w["M"], beta=w["beta"], nprime=w["nprime"], source_block=w["source_block"],
                     basis_max_bytes=w["basis_max_bytes"]),
          "8": dict(N=w8["N"], M=w8["M"], beta=w8["beta"], nprime=w8["nprime"]),
          "4": dict(N=16, M=8, beta=0.3, nprime=14)}
    out = {"requests": len(plan), "arrivals": f"Poisson, mean {SERVING_LARGE['rate_per_s']}/s, seed {seed}",
           "budget_bytes": SERVING_LARGE["budget_bytes"],
           "mix": "2 on the 16^3x32 headline field (both windows; the positive window), L=8 in blocks of 2; "
                  "3 on the 8^4 field (L=4, N=32); 3 on the 4^4 Haar field (L=3, N=16)"}
    for name, prec in (("plain_fp64", ss.FP64), ("mixed", ss.DF)):
        lats = {"16": ss.create_lattice(w["dims"], w["kappa"], w["bc_t"], precision=prec, stream=stream),
                "8": ss.create_lattice(w8["dims"], w8["kappa"], w8["bc_t"], precision=prec, stream=stream),
                "4": ss.create_lattice(dims4, 0.13, -1, precision=prec, stream=stream)}
        ss.upload_gauge(lats["16"], U3)
        ss.upload_gauge(lats["8"], U8)
        ss.upload_gauge(lats["4"], U4)
        torch.cuda.synchronize()
        srv = ss.Server(memory_budget=int(SERVING_LARGE["budget_bytes"]))
        ids, t0, nxt = [], time.perf_counter(), 0
        while True:
            now = time.perf_counter() - t0
            while nxt < len(plan) and arrive[nxt] <= now:
                key, wins, src = plan[nxt]
                k = dict(kw[key])
                N, M = k.pop("N"), k.pop("M")
                ids.append((key, srv.submit_windows(lats[key], wins, N, M, src, **k)))
                nxt += 1
            q, r, f = srv.counts()
            if nxt == len(plan) and q == 0 and r == 0:
                break
            if r > 0 or q > 0:
                srv.progress(wait=(nxt == len(plan) or arrive[nxt] - now > 0.002))
            else:
                time.sleep(max(0.0, arrive[nxt] - now))
        t_end = time.perf_counter() - t0
        lat_ms, pairs, failed, per = [], 0, 0, {}
        for key, i in ids:
            state, ms = srv.status(i)
            lat_ms.append(ms)
            res = srv.take(i)
            if res.status != ss.OK:
                failed += 1
                continue
            _, _, rs, _ = ss.ss_eigpairs(res, want_vectors=False)
            good = int(np.sum(rs <= RES_TOL))
            pairs += good
            per.setdefault(key, []).append({"latency_ms": ms, "eigenpairs": good})
        deferred = srv.deferred()
        srv.close()
        out[name] = {"eigenpairs_per_s": pairs / (t_end - arrive[0]), "eigenpairs": pairs, "failed": failed,
                     "waited_on_memory": deferred, "span_s": t_end - arrive[0],
                     "latency_ms": {"p50": float(np.percentile(lat_ms, 50)), "p99": float(np.percentile(lat_ms, 99))},
                     "per_lattice": per}
        del lats
    out["mixed_vs_plain"] = out["mixed"]["eigenpairs_per_s"] / out["plain_fp64"]["eigenpairs_per_s"]
    return out


def cpu_baseline(budget_s=20.0, gpu_iterations=None, pairs=48, sample_iters=None):
    """The oracle on the host cores, timed on a bounded sample of the
    headline workload and scaled to one step:
      * shifted-CG iterations of source 0 with all 64 shifts (oracle.shifted_cg
        capped at a few iterations) -> seconds per iteration, times the
        iterations of the oracle's own run of this workload (golden file; the
        GPU run's count only when the golden file is absent, and then said)
        times L sources;
      * the moment sums of one window (oracle.moments, 32 solutions, M = 16)
        -> times windows x L;
      * one Rayleigh-Ritz pass (oracle.rayleigh_ritz) on an n x 8 block ->
        its two applications of A scaled to M L = 128 columns and its SVD /
        products by (128 / 8)^2, times the windows."""
    import synthetic
    from oracle import contour, moments, rayleigh_ritz, shifted_cg, wilson
    w = WORKLOAD
    U, src = make_inputs(0)
    dims = w["dims"]
    V = synthetic.volume(dims)
    n = 12 * V
    A = lambda x: wilson.apply_H(U, x, w["kappa"], dims, w["bc_t"])
    z, zeta, wts = [], [], []
    for a, b in w["windows"]:
        gamma, rho = contour.window_from_interval(a, b, w["N"], w["nprime"])
        zz = contour.line_nodes(gamma, rho, w["beta"], w["N"])
        z.append(zz)
        zeta.append(contour.normalise(zz, gamma, rho))
        wts.append(contour.weights_closed_form(zeta[-1]))
    z = np.concatenate(z)
    t0 = time.perf_counter()
    k_cal = 1
    try:
        shifted_cg.shifted_cg(A, src[0], z, tol=w["tol"], max_iter=k_cal)
    except shifted_cg.NoConvergence:
        pass
    t_cal = time.perf_counter() - t0
    k = sample_iters or max(2, min(8, int(0.35 * budget_s / max(t_cal, 1e-6))))
    t0 = time.perf_counter()
    try:
        shifted_cg.shifted_cg(A, src[0], z, tol=w["tol"], max_iter=k)
    except shifted_cg.NoConvergence:
        pass
    t_iter = (time.perf_counter() - t0) / k
    g = synthetic.rng(7)
    y = g.standard_normal((w["N"], V, 4, 3)) + 1j * g.standard_normal((w["N"], V, 4, 3))
    t0 = time.perf_counter()
    moments.moments(y, wts[0], zeta[0], w["M"])
    t_mom = time.perf_counter() - t0
    del y
    m_s, m = 8, w["M"] * w["L"]
    S = g.standard_normal((n, m_s)) + 1j * g.standard_normal((n, m_s))
    t_app = [0.0]

    def apply_cols(X):
        t = time.perf_counter()
        out = A(X.T.reshape(X.shape[1], V, 4, 3)).reshape(X.shape[1], -1).T
        t_app[0] += time.perf_counter() - t
        return out

    t0 = time.perf_counter()
    rayleigh_ritz.rayleigh_ritz(apply_cols, S, rank_tol=1e-14)
    t_rr_all = time.perf_counter() - t0
    del S
    t_rr = t_app[0] * (m / m_s) + (t_rr_all - t_app[0]) * (m / m_s) ** 2
    oracle_iters = _oracle_iterations()
    iters = oracle_iters if oracle_iters is not None else gpu_iterations
    if iters is None:
        raise RuntimeError("no iteration count: tests/golden/config3_iterations.json is missing")
    K = len(w["windows"])
    t_step = t_iter * iters * w["L"] + t_mom * K * w["L"] + t_rr * K
    return {"value": pairs / t_step, "unit": UNIT, "cores": int(_host_cores()), "kind": "oracle",
            "sample": (f"{k} oracle shifted-CG iterations of source 0 with all {len(z)} shifts "
                       f"({t_iter:.2f} s/iteration), the moment sums of one window ({t_mom:.2f} s) and one "
                       f"Rayleigh-Ritz pass on an n x {m_s} block ({t_rr_all:.1f} s; {t_rr:.0f} s scaled to "
                       f"{m} columns); scaled to {iters} iterations x {w['L']} sources, {K} windows = "
                       f"{t_step:.0f} s per step for {pairs} eigenpairs"),
            "iterations_from": ("the oracle's own run (tests/golden/config3_iterations.json)"
                                if oracle_iters is not None else "the GPU run (no oracle count recorded)"),
            "extrapolated": True}


def config1_full():
    """The 4^4 workload of the oracle tests (Haar links, kappa 0.13, L = 3,
    N = 16, M = 8, N' = 14, beta 0.3, [0.374, 0.3930]) solved end to end by
    the oracle on the host: eigenpairs at residual <= 1e-8 per second."""
    import synthetic
    from oracle import ss as oss
    dims = (4, 4, 4, 4)
    U = synthetic.gauge_field(dims, "haar", seed=1)
    src = synthetic.gaussian_sources(dims, 3, seed=100)
    t0 = time.perf_counter()
    out = oss.ss_solve(U, dims, 0.13, -1, (0.374, 0.3930), 16, 8, src, beta=0.3, Nprime=14)
    dt = time.perf_counter() - t0
    pairs = int(np.sum(np.asarray(out["residuals"]) <= RES_TOL))
    return {"eigenpairs": pairs, "seconds": dt, "value": pairs / dt, "unit": UNIT,
            "workload": "4^4 Haar kappa=0.13 L=3 N=16 M=8 beta=0.3 [0.374,0.3930], full oracle solve"}


def run_reference(args):
    world, rank, local = _dist()
    if rank != 0:
        return
    if _oracle_iterations() is None:
        print(json.dumps({"impl": "reference", "unavailable": "the oracle's iteration count of this workload "
                          "(tests/golden/config3_iterations.json) is missing"}), flush=True)
        return
    vals = []
    for i in range(args.warmup + args.steps):
        cb = cpu_baseline(budget_s=args.cpu_budget / 2, sample_iters=2)
        if i >= args.warmup:
            vals.append(cb)
    value = float(np.mean([v["value"] for v in vals]))
    w = WORKLOAD
    c1 = config1_full()
    out = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * 48 / value,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic (seeded smooth SU(3) links, Gaussian sources)",
        "config": {"workload": w["name"], "lattice": list(w["dims"]), "kappa": w["kappa"],
                   "sources": w["L"], "source_block": w["source_block"], "windows": [list(x) for x in w["windows"]],
                   "quad_points_per_window": w["N"], "shifts": w["N"] * len(w["windows"]), "moments": w["M"],
                   "beta": w["beta"], "nprime": w["nprime"], "tol": w["tol"],
                   "parallelism": "host cores (numpy oracle)"},
        "cpu_baseline": {"kind": "oracle", "cores": vals[-1]["cores"], "sample": vals[-1]["sample"], "value": value,
                         "iterations_from": vals[-1]["iterations_from"], "extrapolated": True},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "config1_full_solve": c1,
        "ms_per_step_note": "the extrapolated full step of the oracle on this workload; each of the "
                            f"{args.warmup + args.steps} steps of this run timed a bounded sample of it (about "
                            f"{args.cpu_budget / 2:.0f} s of host work)",
    }
    print(json.dumps(out), flush=True)


BETA_STUDY = (0.2, 0.3, 0.45, 0.6, 0.8, 1.0)


def run_beta_study(ss, stream, big=False):
    """Section 3 leaves the line pair's half gap beta to the user: a larger
    beta moves the points away from the real axis (fewer iterations) and
    flattens the filter (Fig. 2), a smaller one sharpens it (Section 4:
    accuracy up, cost up).  For each beta: seed iterations, accepted pairs,
    pairs at residual <= 1e-8, the largest residual among those, and
    eigenpairs/s (device time of one solve after one warm-up solve), in the
    default stored-residual form.  Workload: the 8^4 one (default) or the
    16^3 x 32 headline (big)."""
    import torch
    w = WORKLOAD if big else CONFIG2
    U, src = make_inputs(0, w)
    lat = ss.create_lattice(w["dims"], w["kappa"], w["bc_t"], stream=stream)
    ss.upload_gauge(lat, torch.from_numpy(U).cuda())
    src_d = torch.from_numpy(src).cuda()
    rows = []
    for beta in BETA_STUDY:
        wb = dict(w, beta=beta)

        def step():
            if big:
                return windows_step(ss, lat, src_d, wb)
            res = ss.ss_solve(lat, wb["interval"], wb["N"], wb["M"], src_d, beta=beta, nprime=wb["nprime"],
                              tol=wb["tol"])
            if res.status != ss.OK:
                raise RuntimeError(res.error)
            ev, _, rs, st = ss.ss_eigpairs(res, want_vectors=False)
            return ev, rs, st

        step()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record(stream)
        ev, rs, st = step()
        e1.record(stream)
        e1.synchronize()
        ms = e0.elapsed_time(e1)
        good = rs <= RES_TOL
        rows.append({"beta": beta, "iterations": st["iterations"], "accepted": int(len(rs)),
                     "converged": int(good.sum()),
                     "max_converged_residual": float(rs[good].max()) if good.any() else None,
                     "ms": ms, "eigenpairs_per_s": float(good.sum()) / (ms / 1e3)})
    return {"workload": w["name"], "rows": rows}


# 48 requests over three lattice sizes (the batched workload): seeded smooth
# fields, each lattice's lowest positive eigenvalue cluster (12 eigenvalues,
# located with the solver on a tiled scan of [0.03, 0.15]); a request with
# L = 1 takes one of three sub-windows of its cluster (3-5 eigenvalues, ends
# in gaps), L = 4 or 8 the whole cluster.
BATCHED = dict(
    lattices={
        "8": dict(dims=(8, 8, 8, 8), kappa=0.125, eps=0.3, seed=2, full=(0.105, 0.120),
                  subs=((0.1095, 0.1123), (0.1123, 0.1146), (0.1146, 0.1170))),
        "12": dict(dims=(12, 12, 12, 12), kappa=0.13, eps=0.4, seed=5, full=(0.0850, 0.0915),
                   subs=((0.0855, 0.0877), (0.0877, 0.08868), (0.08868, 0.0910))),
        "16": dict(dims=(16, 16, 16, 16), kappa=0.135, eps=0.5, seed=6, full=(0.0885, 0.0940),
                   subs=((0.0895, 0.09108), (0.09108, 0.09164), (0.09164, 0.0930))),
    },
    n_requests=48, sources=(1, 4, 8), points=(16, 32, 64), M=8, beta=0.3, nprime={16: 10, 32: 20, 64: 40},
    budget_bytes=200e9, solo_checks=6,
)


def batched_plan(n_requests, seed=29):
    """The request list of the batched workload: (lattice key, interval, N, L,
    source seed, source_block, basis_max_bytes), lattices in turn, L and N
    drawn (seeded)."""
    rng = np.random.default_rng(seed)
    keys = list(BATCHED["lattices"])
    plan = []
    for i in range(n_requests):
        key = keys[i % len(keys)]
        lt = BATCHED["lattices"][key]
        L = int(rng.choice(BATCHED["sources"]))
        N = int(rng.choice(BATCHED["points"]))
        iv = lt["subs"][int(rng.integers(3))] if L == 1 else lt["full"]
        # stored residuals: ~1000 / 1300 / 5000 iterations of 0.8 / 4.0 / 12.6 MB
        # a source on 8^4 / 12^4 / 16^4; the 16^4 runs go one source at a time
        # (63 GB each), and the caps keep every run in the stored-residual form
        sb = 1 if key == "16" and L > 1 else 0
        cap = {"8": 0.0, "12": 6e9 * L, "16": 70e9}[key]
        plan.append((key, iv, N, L, 7000 + i, sb, cap))
    return plan


def run_batched_uneven(ss, stream, n_requests=None, solo_checks=None):
    """The batched workload through the request scheduler: all requests
    submitted at once, each on its own stream with its own CUDA graphs, under
    a 200 GB memory budget; FP64 and float-float lattices.  Reports
    eigenpairs/s at residual <= 1e-8 over the span, p50/p99 latency and the
    requests that waited on memory, and checks that the first few requests'
    eigenvalues equal their solo runs (one request at a time) bit for bit."""
    import torch

    import synthetic
    cfg = BATCHED
    n_requests = cfg["n_requests"] if n_requests is None else n_requests
    solo_checks = cfg["solo_checks"] if solo_checks is None else solo_checks
    plan = batched_plan(n_requests)
    fields = {k: synthetic.gauge_field(v["dims"], "smooth", seed=v["seed"], eps=v["eps"])
              for k, v in cfg["lattices"].items()}
    out = {"requests": n_requests, "arrivals": "all at once",
           "mix": "8^4 (kappa 0.125, eps 0.3), 12^4 (0.13, 0.4), 16^4 (0.135, 0.5) in turn; L in {1, 4, 8}, "
                  "N in {16, 32, 64}, M 8; L = 1 on a 3-5 eigenvalue sub-window, else the 12-eigenvalue cluster",
           "budget_bytes": cfg["budget_bytes"],
           "launch": "per-request streams and CUDA graphs through the scheduler (no single launch across "
                     "lattices)"}

    def submit(srv, lats, item):
        key, iv, N, L, sseed, sb, cap = item
        lt = cfg["lattices"][key]
        src = torch.from_numpy(synthetic.gaussian_sources(lt["dims"], L, seed=sseed)).cuda()
        return srv.submit_windows(lats[key], [iv], N, cfg["M"], src, beta=cfg["beta"], nprime=cfg["nprime"][N],
                                  source_block=sb, basis_max_bytes=cap)

    def serve(lats, items):
        srv = ss.Server(int(cfg["budget_bytes"]))
        t0 = time.perf_counter()
        ids = [submit(srv, lats, it) for it in items]
        while True:
            q, r, f = srv.counts()
            if q == 0 and r == 0:
                break
            srv.progress(wait=True)
        span = time.perf_counter() - t0
        lat_ms, pairs, failed, evs = [], 0, 0, []
        for i in ids:
            _, ms = srv.status(i)
            lat_ms.append(ms)
            res = srv.take(i)
            if res.status != ss.OK:
                failed += 1
                evs.append(None)
                continue
            ev, _, rs, _ = ss.ss_eigpairs(res, want_vectors=False)
            pairs += int(np.sum(rs <= RES_TOL))
            evs.append((ev, rs))
        deferred = srv.deferred()
        srv.close()
        return {"eigenpairs_per_s": pairs / span, "eigenpairs": pairs, "failed": failed,
                "waited_on_memory": deferred, "span_s": span,
                "latency_ms": {"p50": float(np.percentile(lat_ms, 50)), "p99": float(np.percentile(lat_ms, 99))}}, evs

    for name, prec in (("plain_fp64", ss.FP64), ("mixed", ss.DF)):
        lats = {}
        for k, v in cfg["lattices"].items():
            lats[k] = ss.create_lattice(v["dims"], v["kappa"], -1, precision=prec, stream=stream)
            ss.upload_gauge(lats[k], fields[k])
        res, evs = serve(lats, plan)
        same = 0
        for j in range(min(solo_checks, len(plan))):
            _, evs1 = serve(lats, [plan[j]])
            a, b = evs[j], evs1[0]
            same += int(a is not None and b is not None and np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]))
        res["solo_identical"] = f"{same} of {min(solo_checks, len(plan))}"
        out[name] = res
        del lats
    out["mixed_vs_plain"] = out["mixed"]["eigenpairs_per_s"] / out["plain_fp64"]["eigenpairs_per_s"]
    return out


def run_only(args):
    """One secondary leg alone (the commands of the committed ncu captures)."""
    import torch

    import paper_1004_0292_gb300 as ss
    from paper_1004_0292_gb300 import build as ssbuild
    ssbuild.build()
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    peaks = _measured_peaks()
    if args.only == "stencil_large":
        ss.set_stencil_variant(args.stencil_variant)
        out = run_stencil_large(ss, stream, peaks, rhs=args.stencil_rhs)
    elif args.only == "batched_uneven":
        out = run_batched_uneven(ss, stream)
    elif args.only.startswith("beta_study"):
        out = run_beta_study(ss, stream, big=args.only.endswith("16x32"))
    else:
        flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")
        out = run_config2(ss, stream, flush, args, 1, peaks)
    print(json.dumps({"only": args.only, "result": out}), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-mixed", action="store_true", help="skip the float-float arm")
    ap.add_argument("--no-serving", action="store_true", help="skip the request-scheduler run")
    ap.add_argument("--no-update-form", action="store_true", help="skip the shift-vector update form")
    ap.add_argument("--no-config2", action="store_true", help="skip the 8^4 legs")
    ap.add_argument("--no-e2e", action="store_true", help="skip the end-to-end (host buffers) leg")
    ap.add_argument("--e2e-steps", type=int, default=1)
    ap.add_argument("--cpu-budget", type=float, default=30.0)
    ap.add_argument("--stencil-rhs", type=int, default=None, help="right-hand sides of stencil_large (default 8)")
    ap.add_argument("--stencil-variant", type=int, default=-1,
                    help="FP32 stencil variant for stencil_large (0..7; -1: the autotuner's choice)")
    ap.add_argument("--only", choices=["stencil_large", "config2", "beta_study", "beta_study_16x32", "batched_uneven"],
                    default=None,
                    help="run one secondary leg alone and print its JSON (profiling runs)")
    args = ap.parse_args()
    if args.only is not None:
        run_only(args)
        return
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
