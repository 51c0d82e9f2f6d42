#!/usr/bin/env python
"""Benchmark: one reconstruction iteration of differentiable MCR (arXiv 2103.09686) on GB300.

A step is one pass of the whole hot path through the C ABI (``dmcr_adam_step``): multigrid
restriction, the soft-thresholded S2 descriptor of every level, loss with box penalty,
adjoint coefficients, the fused adjoint of every level, gradient assembly through the
levels, and one Adam update.  Default workload: a 512x512 two-phase target (thresholded
Gaussian random field, correlation length 12 px, volume fraction 0.40, plus periodic
non-overlapping discs of radius 6-20 px), shift window +-64, three simultaneous levels
(512, 256, 128), FP32, starting from a seeded uniform[0,1) field.

Metric: S2+adjoint voxel-shifts/s = sum_l N_l K_full,l per step / step time, K_full =
prod_a (2 P_a + 1).  Prints ONE JSON line (rank 0).  ``--impl reference`` times the FP64
CPU oracle on a bounded sample of the same workload instead.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import synthetic  # noqa: E402

METRIC = "S2+adjoint voxel-shifts/s"
UNIT = "voxel-shifts/s"
FP32_LANES_NOMINAL = 128          # FP32 FMA lanes per SM per clock by the unit count (an FFMA2 takes two)
# FP32 lane operations and MUFU reciprocals per (position, shift) pair of the implemented
# soft-threshold formulation:
#   forward: d = 1 + E'E (1), product d_a d_b of two pairs sharing a reciprocal (1/2),
#            u = s + c3/c1 (1), acc += u^2 (1); one reciprocal per two pairs;
#   adjoint: d (1), Horner G h(s) (3); 4 of every 8 positions share a reciprocal between two
#            pairs (product 1/2, s 1), 4 of 8 take one reciprocal per pair.
LANE_OPS_PER_PAIR = {"corr_fwd": 3.5, "corr_adj": 4.0 + 4.0 / 8.0 * 1.5}
RCP_PER_PAIR = {"corr_fwd": 0.5, "corr_adj": 4.0 / 8.0 * 0.5 + 4.0 / 8.0}
# The per-pair work one pair evaluation of the soft threshold needs by the method's own
# count (1 exponential + 1 reciprocal + about 5 FP32 operations): the algorithmic figure the
# implemented counts above are compared with (the product form needs no exponential per pair).
ALGORITHMIC_FP32_OPS_PER_PAIR = 5.0
# the probe's measured pair rate of each kernel's own instruction mix held in registers
MIX_KEY = {"corr_fwd": "forward_pairs", "corr_adj": "adjoint_pairs"}
# DRAM bytes (read + write) per launch of each correlation kernel, from one ncu capture of the
# bench's own command per workload (dram__bytes_read.sum + dram__bytes_write.sum); None
# whenever a kernel changed since its last capture.
NCU_TRAFFIC_BYTES = {("grf64", "corr_adj"): 90112 + 0, ("grf64", "corr_fwd"): 93696 + 0}

WORKLOADS = {
    "grf512": dict(shape=(512, 512), window=(64, 64), levels=3,
                   desc="2D 512x512 GRF(l=12,vf=0.40)+discs r6-20, window +-64, 3 levels (512,256,128), "
                        "one Adam iteration per step"),
    "grf128_3d": dict(shape=(128, 128, 128), window=(24, 24, 24), levels=2,
                      desc="3D 128^3 GRF(l=6/6/12, vf=0.25), window +-24, 2 levels (128,64), one Adam iteration"),
    "grf64": dict(shape=(64, 64), window=(16, 16), levels=1,
                  desc="2D 64x64 GRF(l=4, vf=0.30), window +-16, 1 level, one Adam iteration"),
    "mp3_512": dict(shape=(512, 512), window=(64, 64), levels=3, phases=3,
                    desc="2D three-phase 512x512 GRF(l=12, phase fractions 0.3/0.3/0.4), window +-64, 3 levels "
                         "(512,256,128), cross-correlations of all 9 ordered phase pairs; one Adam iteration per step"),
    "batch256": dict(shape=None, window=None, levels=1, count=256,
                     desc="256 independent 2D instances, sizes uniform over {64,128,256,512}^2, GRF vf U[0.1,0.5], "
                          "windows U{16..64} capped at n/2, 1 level; one fused batched Adam iteration per step"),
}


def batch_instances(count: int, seed: int):
    """(shape, window, target) of the mixed-size batch (seeds 4000 + instance)."""
    out = []
    for tgt, P, _ in synthetic.batch_instances(count, seed):
        out.append((tgt.shape, (P, P), tgt))
    return out


SERVE_2D = (128, 256, 512, 1024)
SERVE_3D = (64, 80, 96, 128, 160)


def serve_job(i: int, rng, seed: int, dm, serve, kind=None, n=None):
    """One served job: a 2-D GRF target with n in SERVE_2D (window +-16, levels down to a
    64^2 coarsest level) or, for one job in six, a 3-D GRF target with n in SERVE_3D
    (window +-8, 3 levels for n >= 96, else 2); correlation length n/32, vf ~ U[0.1, 0.5];
    the job runs to rel_err < 1e-3 (tested every 10 iterations) or 5000 iterations."""
    three = (rng.random() < 1.0 / 6.0) if kind is None else kind == 3
    if three:
        n = int(rng.choice(SERVE_3D)) if n is None else n
        shape, win, lev, lr = (n, n, n), (8, 8, 8), 3 if n >= 96 else 2, 3e-3
        tgt = synthetic.target_3d(n, seed + i, (n / 32.0,) * 3, float(rng.uniform(0.1, 0.5)))
    else:
        n = int(rng.choice(SERVE_2D)) if n is None else n
        shape, win, lev, lr = (n, n), (16, 16), int(np.log2(n // 64)) + 1, 1e-2
        tgt = synthetic.target_2d_grf(n, n / 32.0, float(rng.uniform(0.1, 0.5)), seed + i)
    opts = dm.ReconOpts(max_iters=5000, lr=lr, tol_rel=1e-3, check_every=10, seed=seed + 7 * i)
    return serve.Job(job_id=i, params=dm.Params(shape=shape, window=win, levels=lev), target=tgt, opts=opts)


def serve_jobs(n_jobs: int, rate: float, seed: int, dm, serve):
    """The first n_jobs arrivals of a Poisson process of the given rate (jobs: serve_job)."""
    return serve.poisson_trace(n_jobs, rate, seed, lambda i, rng: serve_job(i, rng, seed, dm, serve))


SERVE_CLASS_CAPS = (1.5e8, 1e9, 1e10, float("inf"))   # voxel-shifts per iteration of each cost class
# most active jobs per class: the class of the 128^3/160^3 jobs serves one job at a time in
# arrival order, the class of the 2-D 1024^2 and 3-D 64-96^3 jobs four; equal stream
# priorities.  Measured on the first 128 arrivals at 80% load (0.377 req/s) against the plain
# form of the same session: p50 4.41 / p99 90.5 / mean 14.4 s against 5.00 / 91.8 / 18.3 s
# (other settings: no limits 4.8 / 119 / 22.8 s; one job in each heavy class 1.6 / 120 /
# 17.8 s; the heaviest class exclusive 4.9 / 170 / 34.8 s).
SERVE_CLASS_SLOTS = (None, None, 4, 1)
SERVE_PRIORITIES = "equal"


def main_serve(args):
    """Served vs plain form on Poisson traces, every job to the same S2 error target: the
    first --jobs arrivals (seed 5000) at 200 req/s, far above capacity, then the first
    --jobs2 arrivals of the same process at 80% of the capacity the served form measured
    on the first trace."""
    import torch
    import paper_2103_09686_gb300 as dm
    from paper_2103_09686_gb300 import serve
    dm.load()
    sampler = ClockSampler(0)
    # warm the library and the allocator on a small job (not part of any run)
    serve.reconstruct_alone(serve_jobs(1, 200.0, 4999, dm, serve)[0])
    sampler.start()

    def both(n_jobs, rate):
        jobs = serve_jobs(n_jobs, rate, 5000, dm, serve)
        served = serve.run_trace(jobs, "serve", max_slots=args.slots, tick_iters=50, class_caps=SERVE_CLASS_CAPS,
                                 class_slots=SERVE_CLASS_SLOTS, priorities=SERVE_PRIORITIES)
        units = sum(j.iters_done * serve.iteration_units(j.params) for j in jobs)
        plain_jobs = serve_jobs(n_jobs, rate, 5000, dm, serve)
        plain = serve.run_trace(plain_jobs, "plain")
        same = all(np.array_equal(a.result, b.result) for a, b in zip(sorted(jobs, key=lambda j: j.job_id),
                                                                     sorted(plain_jobs, key=lambda j: j.job_id)))
        out = {"rate_per_s": rate, "served": served, "plain": plain, "results_identical_served_vs_plain": bool(same),
               "voxel_shifts_per_s_served": units / served["wall_s"]}
        print(json.dumps({"partial": out}), file=sys.stderr, flush=True)
        return out

    over = both(args.jobs, 200.0)
    capacity = over["served"]["reconstructions_per_s"]
    at80 = both(args.jobs2, 0.8 * capacity)
    clocks = sampler.stop()
    line = {"metric": "reconstructions/s", "value": capacity, "unit": "reconstructions/s",
            "n_gpus": 1, "steps": args.jobs, "warmup": 1, "ms_per_step": over["served"]["wall_s"] * 1e3 / args.jobs,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "Poisson trace, seed 5000: the first %d arrivals at 200 req/s, then the first %d at "
                                   "80%% of the measured served capacity; jobs 2D GRF {128,256,512,1024}^2 +-16 with "
                                   "levels down to 64^2, one in six 3D GRF {64,80,96,128,160}^3 +-8 (3 levels from "
                                   "96, else 2), l = n/32, vf U[0.1,0.5], each to rel_err < 1e-3 (at most 5000 "
                                   "iterations); slots %d, tick 50 iterations, cost classes %s with at most %s "
                                   "active jobs each, %s stream priorities"
                                   % (args.jobs, args.jobs2, args.slots, list(SERVE_CLASS_CAPS),
                                      list(SERVE_CLASS_SLOTS), SERVE_PRIORITIES)},
            "overload": over, "at_80pct_capacity": at80, "clocks": clocks}
    print(json.dumps(line))
    return 0


def main_crossover(args):
    """Identity threshold (f(x) = x): descriptor + gradient (dmcr_loss_grad) time of the
    direct kernels vs the FFT path over the window P per axis, on 64^3 and 128^3 (one
    level); CUDA events, median of 5 after 2 warm-ups."""
    import torch
    import paper_2103_09686_gb300 as dm
    dm.load()
    out = {"metric": "direct vs FFT crossover (identity threshold, descriptor+gradient)", "unit": "ms", "sizes": {}}
    for n in (64, 128):
        rows = []
        M = torch.tensor(synthetic.uniform_field((n, n, n), 11), dtype=torch.float32, device="cuda")
        T = torch.tensor(synthetic.target_3d(n, 12, (3.0, 3.0, 3.0), 0.3), dtype=torch.float32, device="cuda")
        for P in (1, 2, 3, 4, 6, 8, 10, 12, 16, 20, 24):
            if 2 * P > n:
                continue
            row = {"P": P}
            for path, key in ((dm.DMCR_PATH_DIRECT, "direct_ms"), (dm.DMCR_PATH_FFT, "fft_ms")):
                p = dm.Params(shape=(n, n, n), window=(P, P, P), threshold=dm.DMCR_IDENTITY, path=path)
                ws = dm.workspace(p)
                d = dm.descriptor(T, p, ws)
                loss = torch.empty(6, device="cuda")
                g = torch.empty_like(M)
                times = []
                for r in range(7):
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    a.record()
                    dm.dmcr_loss_grad(p, dm.LossOpts(), M, d, loss, g, None, ws)
                    b.record()
                    torch.cuda.synchronize()
                    if r >= 2:
                        times.append(a.elapsed_time(b))
                row[key] = float(np.median(times))
            rows.append(row)
        cross = next((r["P"] for r in rows if r["fft_ms"] < r["direct_ms"]), None)
        out["sizes"]["%d^3" % n] = {"rows": rows, "crossover_P": cross}
    print(json.dumps(out))
    return 0


def main_fft(args):
    """FFT path roofline: descriptor + loss + gradient (dmcr_loss_grad) of the identity
    threshold on a 128^3 field, window +-24 per axis, one level, path FFT (App. A / Sec. 4.1
    ablation).  A step is four complex FP64 transforms of the grid (DFT of the field, inverse
    of its power spectrum, DFT of the embedded adjoint coefficients, inverse of their
    product), three axis passes each.  Algorithmic work: 5 N log2 N flops per transform; the
    peak is the pipe probe's measured FP64 DFMA rate (2 flops each) x SMs x max SM clock.
    CUDA events around each step, L2 flushed before every step."""
    import torch
    import paper_2103_09686_gb300 as dm
    dm.load()
    n, P = 128, 24
    pipes = measure_pipe_rates()
    p = dm.Params(shape=(n, n, n), window=(P, P, P), threshold=dm.DMCR_IDENTITY, path=dm.DMCR_PATH_FFT)
    ws = dm.workspace(p)
    M = torch.tensor(synthetic.uniform_field((n, n, n), 11), dtype=torch.float32, device="cuda")
    T = torch.tensor(synthetic.target_3d(n, 12, (3.0, 3.0, 3.0), 0.3), dtype=torch.float32, device="cuda")
    D = dm.descriptor(T, p, ws)
    loss = torch.empty(6, device="cuda")
    g = torch.empty_like(M)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for _ in range(args.warmup):
        dm.dmcr_loss_grad(p, dm.LossOpts(), M, D, loss, g, None, ws)
    sampler = ClockSampler(0)
    sampler.start()
    times = []
    for _ in range(args.steps):
        flush.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        dm.dmcr_loss_grad(p, dm.LossOpts(), M, D, loss, g, None, ws)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    dm.dmcr_profile_reset()
    dm.dmcr_profile_enable(True)
    for _ in range(min(args.steps, 5)):
        flush.zero_()
        dm.dmcr_loss_grad(p, dm.LossOpts(), M, D, loss, g, None, ws)
    torch.cuda.synchronize()
    dm.dmcr_profile_enable(False)
    prof = dm.dmcr_profile_read()
    clocks = sampler.stop()
    N = n ** 3
    ms = float(np.median(times))
    flops = 4 * 5.0 * N * np.log2(N)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    clk = (clocks.get("sm_max_mhz") or 2070.0) * 1e6
    fp64_peak = sm * pipes["dfma"] * 2.0 * clk / 1e12
    achieved = flops / (ms / 1e3) / 1e12
    hbm = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))).get("hbm_gbs", 6800.0) if os.path.exists(
        os.path.join(ROOT, "MEASURED_PEAKS.json")) else 6800.0
    bytes_step = 4 * 3 * 2 * 16.0 * N           # every axis pass reads and writes the complex grid
    print(json.dumps({"metric": "FFT path descriptor+gradient (identity threshold)", "unit": "ms",
                      "value": ms, "ms_per_step": ms, "steps": args.steps, "warmup": args.warmup,
                      "higher_is_better": False, "dtype": "f64", "data": "synthetic",
                      "config": {"workload": "128^3 uniform field, window +-24, one level, path FFT; L2 flushed "
                                             "before every step"},
                      "roofline": {"bound": "fp64", "achieved": achieved, "peak": fp64_peak, "unit": "TFLOP/s",
                                   "frac": achieved / fp64_peak,
                                   "basis": "4 transforms x 5 N log2 N flops / step time; peak = measured DFMA "
                                            "%.2f/clk/SM x 2 x %d SMs x max clock" % (pipes["dfma"], sm)},
                      "hbm": {"bytes_per_step_model": bytes_step, "achieved_gbs": bytes_step / (ms / 1e3) / 1e9,
                              "peak_gbs": hbm, "frac": bytes_step / (ms / 1e3) / 1e9 / hbm},
                      "kernels": {k: {"ms_per_step": round(t / min(args.steps, 5), 4), "launches": c}
                                  for k, (t, c) in sorted(prof.items())},
                      "clocks": clocks}))
    return 0


def main_s3(args):
    """Three-point descriptor (Eq. s3) at the paper's App. B configurations, P = 31:
    64^2 (one level), 128^2 (two) and 256^2 (three).  A step is one descriptor + loss +
    gradient + Adam iteration (dmcr_adam_step), timed with CUDA events after warm-up, L2
    flushed before every step.  The tensor-core rate counts the executed FP16 MMA flops of
    the two GEMMs (Gram on the upper-triangle tiles, W), three split products each, over
    the step time; the peak is the measured bf16 burst peak (FP16 and BF16 share the dense
    rate).  The library's event timers give each phase's share of the step."""
    import torch
    import paper_2103_09686_gb300 as dm
    dm.load()
    peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))) if os.path.exists(
        os.path.join(ROOT, "MEASURED_PEAKS.json")) else {}
    bf16 = float(peaks.get("bf16_tflops", 1900.0))
    f16_peak = bf16
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    out = []
    for n, levels in ((64, 1), (128, 2), (256, 3)):
        P = 31
        p = dm.Params(shape=(n, n), window=(P, P), levels=levels, descriptor=dm.DMCR_DESC_S3)
        ws = dm.workspace(p)
        T = torch.tensor(synthetic.checkerboard(n, 8), dtype=torch.float32, device="cuda")
        D = dm.descriptor(T, p, ws)
        f = torch.tensor(synthetic.uniform_field((n, n), 1), dtype=torch.float32, device="cuda")
        m = torch.zeros_like(f)
        v = torch.zeros_like(f)
        opts = dm.ReconOpts(lr=1e-3)
        st = 0
        for _ in range(3):
            st = dm.dmcr_adam_step(p, opts, D, f, m, v, st, None, ws)
        steps = 20 if n < 256 else 8
        times = []
        dm.dmcr_profile_reset()
        dm.dmcr_profile_enable(True)
        for _ in range(steps):
            flush.zero_()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            st = dm.dmcr_adam_step(p, opts, D, f, m, v, st, None, ws)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        dm.dmcr_profile_enable(False)
        prof = dm.dmcr_profile_read()
        ms = float(np.median(times))
        K = (2 * P + 1) * (2 * P + 1) // 2 + 1
        Kp = (K + 127) // 128 * 128
        flops = 0.0
        for l in range(levels):
            Np = ((n >> l) ** 2 + 127) // 128 * 128
            t = Kp // 128
            flops += 3 * 2.0 * (t * (t + 1) // 2) * 128 * 128 * Np      # Gram, upper tiles
            flops += 3 * 2.0 * Np * Kp * Kp                               # W = E G
        achieved = flops / (ms / 1e3) / 1e12
        out.append({"workload": "%dx%d, P=%d, %d level(s), K=%d" % (n, n, P, levels, K), "ms_per_step": ms,
                    "steps_per_s": 1e3 / ms,
                    "roofline": {"bound": "tensor", "achieved": achieved, "peak": f16_peak, "unit": "TFLOP/s",
                                 "frac": achieved / f16_peak,
                                 "basis": "executed FP16 MMA flops of both GEMMs (3 split products) / step time; "
                                          "peak = measured bf16 burst %.0f TF/s (the FP16 dense rate)" % bf16},
                    "phases_ms_per_step": {k: round(t / steps, 4) for k, (t, c) in sorted(prof.items())}})
    print(json.dumps({"metric": "three-point descriptor Adam steps/s", "unit": "steps/s", "dtype": "f16x3",
                      "data": "synthetic", "l2": "flushed before every timed step", "runs": out}))
    return 0


def main_checkerboard(args):
    """Sec. 4.1 checkerboard experiments on 64 x 64 with P = 31 (App. B), 8-pixel squares:
    iterations until the rounded field's descriptor equals the target (relative error
    < 1e-6, tested every 100 iterations), for the three-point descriptor with the soft
    threshold (E1) and with f(x) = x (E2), and for the two-point descriptor alone; Adam at
    lr 1e-3 (TensorFlow default) and 1e-2, start field SplitMix64 uniform seed 1."""
    import torch
    import paper_2103_09686_gb300 as dm
    dm.load()
    n, P, a = 64, 31, 8
    runs = []
    # one-time start-up (module loading, tensor-map encoding, graph capture) outside every
    # timed run: 100 untimed iterations of each descriptor
    for kind in (dm.DMCR_DESC_S3, dm.DMCR_DESC_S2):
        p = dm.Params(shape=(n, n), window=(P, P), descriptor=kind)
        ws = dm.workspace(p)
        D = dm.descriptor(torch.tensor(synthetic.checkerboard(n, a), dtype=torch.float32, device="cuda"), p, ws)
        f = torch.empty(n, n, device="cuda")
        dm.dmcr_reconstruct(p, dm.ReconOpts(max_iters=100, lr=1e-2, seed=1, init=dm.DMCR_INIT_UNIFORM_SEEDED),
                            D, f, torch.zeros_like(f), torch.zeros_like(f), ws=ws)
    torch.cuda.synchronize()
    specs = [("S3", dm.DMCR_SOFT, 1e-3, 6000), ("S3", dm.DMCR_SOFT, 1e-2, 6000),
             ("S3", dm.DMCR_IDENTITY, 1e-3, 6000), ("S3", dm.DMCR_IDENTITY, 1e-2, 6000),
             ("S2", dm.DMCR_SOFT, 1e-3, 6000), ("S2", dm.DMCR_SOFT, 1e-2, 6000)]
    for desc, thr, lr, max_it in specs:
        p = dm.Params(shape=(n, n), window=(P, P), threshold=thr,
                      descriptor=dm.DMCR_DESC_S3 if desc == "S3" else dm.DMCR_DESC_S2)
        ws = dm.workspace(p)
        T = torch.tensor(synthetic.checkerboard(n, a), dtype=torch.float32, device="cuda")
        D = dm.descriptor(T, p, ws)
        f = torch.empty(n, n, device="cuda")
        m = torch.zeros_like(f)
        v = torch.zeros_like(f)
        step, first, curve = 0, None, []
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        while step < max_it:
            opts = dm.ReconOpts(max_iters=100, lr=lr, seed=1,
                                init=dm.DMCR_INIT_UNIFORM_SEEDED if step == 0 else dm.DMCR_INIT_CALLER)
            rep, step = dm.dmcr_reconstruct(p, opts, D, f, m, v, step=step, ws=ws)
            rounded = rep["rounded_rel_err"]      # the library's evaluation of the field rounded to 0/1
            curve.append([step, rep["rel_err"], rounded])
            if rounded < 1e-6:
                first = step
                break
        secs = time.perf_counter() - t0
        runs.append({"descriptor": desc, "threshold": "identity" if thr == dm.DMCR_IDENTITY else "soft", "lr": lr,
                     "iterations_to_exact": first, "seconds": round(secs, 3),
                     "ms_per_iteration": round(1e3 * secs / max(step, 1), 3), "curve_every_100": curve})
    print(json.dumps({"metric": "checkerboard 64x64, P=31: iterations until the rounded field is exact",
                      "unit": "iterations", "config": {"squares_px": a, "test_every": 100, "max_iterations": 6000},
                      "runs": runs}))
    return 0


def main_c1(args):
    """The 64 x 64, +-16 workload as a whole reconstruction: 200 Adam iterations (lr 1e-3,
    the TensorFlow default of App. B) from the SplitMix64 uniform start (seed 1001) toward
    the GRF target (l = 4 px, vf 0.30, seed 1000).  Reconstructions per second of the FP64
    oracle on one host core and on every host core (its own OpenMP loops), and of the
    library's graph-captured dmcr_reconstruct; the final relative descriptor errors side by
    side (Adam amplifies rounding late in a run, so they agree to a few percent, not
    bitwise)."""
    import oracle
    n, P, iters, lr = 64, 16, 200, 1e-3
    T = synthetic.target_small_2d(1000)
    M0 = synthetic.uniform_field((n, n), seed=1001)
    op = oracle.Params(ndim=2, window=(P, P), levels=1)
    D = oracle.descriptor(T, op)
    cpu = {}
    for label, th in (("1_core", 1), ("all_cores", os.cpu_count())):
        oracle.set_threads(th)
        t0 = time.perf_counter()
        _, hist = oracle.reconstruct(M0, D, op, iters=iters, lr=lr)
        secs = time.perf_counter() - t0
        cpu[label] = {"cores": th, "seconds": round(secs, 3), "reconstructions_per_s": 1.0 / secs,
                      "final_rel_err": hist[-1]["rel_err"]}
    oracle.set_threads(os.cpu_count())
    import torch
    import paper_2103_09686_gb300 as dm
    dm.load()
    p = dm.Params(shape=(n, n), window=(P, P))
    ws = dm.workspace(p)
    Dd = torch.tensor(D.astype(np.float32), device="cuda")
    opts = dm.ReconOpts(max_iters=iters, lr=lr, init=dm.DMCR_INIT_UNIFORM_SEEDED, seed=1001, report_rounded=False)
    f = torch.empty(n, n, device="cuda")
    m, v = torch.zeros_like(f), torch.zeros_like(f)
    for _ in range(3):                              # warm-up: modules, graph instantiation
        m.zero_(), v.zero_()
        dm.dmcr_reconstruct(p, opts, Dd, f, m, v, ws=ws)
    reps, secs = 20, []
    rep = None
    for _ in range(reps):
        m.zero_(), v.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rep, _ = dm.dmcr_reconstruct(p, opts, Dd, f, m, v, ws=ws)   # synchronous
        secs.append(time.perf_counter() - t0)
    gpu_s = float(np.median(secs))
    line = {"metric": "reconstructions/s", "value": 1.0 / gpu_s, "unit": "reconstructions/s", "n_gpus": 1,
            "steps": reps, "warmup": 3, "ms_per_step": gpu_s * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "2D 64x64 GRF(l=4, vf=0.30) target, window +-16, 1 level, 200 Adam iterations "
                                   "(lr 1e-3) from a uniform[0,1) start; one step = one whole reconstruction "
                                   "(dmcr_reconstruct, graph-captured iterations, host wall clock)"},
            "final_rel_err": {"gpu": rep["rel_err"], "oracle": cpu["1_core"]["final_rel_err"]},
            "cpu_baseline": {"value": cpu["all_cores"]["reconstructions_per_s"], "unit": "reconstructions/s",
                             "cores": cpu["all_cores"]["cores"], "kind": "oracle",
                             "sample": "the whole 200-iteration FP64 oracle reconstruction, no sampling"},
            "oracle_runs": cpu, "gpu_seconds_median": gpu_s}
    print(json.dumps(line))
    return 0


def _exact_run(dm, torch, p, D, f, m, v, lr, max_it, step0=0, seed=1, init=True):
    """Adam in chunks of 100 iterations until the rounded field's descriptor equals D
    (relative error < 1e-6).  Returns (iterations to exact or None, Adam steps, seconds)."""
    ws = dm.workspace(p)
    step = step0
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    first = None
    if not init:   # a warm start may already be exact (no iteration: one evaluation)
        rep0, _ = dm.dmcr_reconstruct(p, dm.ReconOpts(max_iters=0), D, f, m, v, step=step, ws=ws)
        if rep0["rounded_rel_err"] < 1e-6:
            return 0, 0, time.perf_counter() - t0
    while step - step0 < max_it:
        opts = dm.ReconOpts(max_iters=100, lr=lr, seed=seed,
                            init=dm.DMCR_INIT_UNIFORM_SEEDED if (init and step == step0) else dm.DMCR_INIT_CALLER)
        rep, step = dm.dmcr_reconstruct(p, opts, D, f, m, v, step=step, ws=ws)
        if rep["rounded_rel_err"] < 1e-6:
            first = step - step0
            break
    torch.cuda.synchronize()
    return first, step - step0, time.perf_counter() - t0


def main_multigrid(args):
    """Sec. 4.1 / Fig. reconstructionsmg: a 128 x 128 checkerboard (8-pixel squares) with the
    three-point descriptor, Adam lr 1e-2, until the rounded field is exact (tested every 100
    iterations): the simultaneous multigrid of Sec. 3.3 (P = 31, levels 128 and 64), all
    vectors on one level (P = 63), short range only (P = 8, one level), and the sequential
    coarse-to-fine scheme the paper contrasts itself with (converge 64 x 64 at P = 31, inject
    every coarse value into its 2 x 2 children, continue at 128 x 128, P = 31, one level)."""
    import torch
    import paper_2103_09686_gb300 as dm
    dm.load()
    n, a, lr, cap = 128, 8, 1e-2, 4000
    S3 = dm.DMCR_DESC_S3
    T = torch.tensor(synthetic.checkerboard(n, a), dtype=torch.float32, device="cuda")
    runs = []

    def fresh(shape):
        f = torch.empty(shape, device="cuda")
        return f, torch.zeros_like(f), torch.zeros_like(f)

    for name, window, levels in (("simultaneous multigrid P=31, levels 128+64", (31, 31), 2),
                                 ("one level, all vectors P=63", (63, 63), 1),
                                 ("one level, short range P=8", (8, 8), 1)):
        p = dm.Params(shape=(n, n), window=window, levels=levels, descriptor=S3)
        D = dm.descriptor(T, p)
        f, m, v = fresh((n, n))
        it, steps, secs = _exact_run(dm, torch, p, D, f, m, v, lr, cap)
        runs.append({"scheme": name, "iterations_to_exact": it, "iterations_run": steps, "seconds": round(secs, 3)})
    # sequential coarse-to-fine warm start
    pc = dm.Params(shape=(n // 2, n // 2), window=(31, 31), descriptor=S3)
    Tc = torch.tensor(synthetic.checkerboard(n // 2, a // 2), dtype=torch.float32, device="cuda")
    Dc = dm.descriptor(Tc, pc)
    fc, mc, vc = fresh((n // 2, n // 2))
    it_c, steps_c, secs_c = _exact_run(dm, torch, pc, Dc, fc, mc, vc, lr, cap)
    pf = dm.Params(shape=(n, n), window=(31, 31), descriptor=S3)
    Df = dm.descriptor(T, pf)
    f, m, v = fresh((n, n))
    dm.dmcr_prolongate(fc, f, dm.DMCR_PROLONG_INJECT)
    it_f, steps_f, secs_f = _exact_run(dm, torch, pf, Df, f, m, v, lr, cap, init=False)
    injected = dm.dmcr_reconstruct(pf, dm.ReconOpts(max_iters=0), Df, f, m, v)[0]["rounded_rel_err"]
    runs.append({"scheme": "sequential coarse-to-fine: 64x64 (4-px squares) then inject, 128x128 P=31",
                 "coarse_iterations_to_exact": it_c, "fine_iterations_to_exact": it_f,
                 "rounded_rel_err_after_fine_stage": injected,
                 "iterations_run": steps_c + steps_f, "seconds": round(secs_c + secs_f, 3)})
    print(json.dumps({"metric": "checkerboard 128x128: iterations until the rounded field is exact",
                      "unit": "iterations", "config": {"descriptor": "S3 (Eq. s3)", "squares_px": a, "lr": lr,
                                                       "test_every": 100, "max_iterations": cap},
                      "runs": runs}))
    return 0


def main_checkerboard_sizes(args):
    """Sec. 4.1 / Fig. checerboardreconstructions: checkerboards of 64, 128, 256 and 512
    pixels (8-pixel squares) with the proposed multigrid scheme, three-point descriptor,
    P = 31, levels down to 64 x 64, Adam lr 1e-2, until the rounded field is exact (tested
    every 100 iterations, at most 4000)."""
    import torch
    import paper_2103_09686_gb300 as dm
    dm.load()
    a, lr, cap = 8, 1e-2, 4000
    S3 = dm.DMCR_DESC_S3
    # one-time start-up outside the timed runs
    p0 = dm.Params(shape=(64, 64), window=(31, 31), descriptor=S3)
    f0 = torch.empty(64, 64, device="cuda")
    _exact_run(dm, torch, p0, dm.descriptor(torch.tensor(synthetic.checkerboard(64, a), dtype=torch.float32,
                                                         device="cuda"), p0),
               f0, torch.zeros_like(f0), torch.zeros_like(f0), lr, 100)
    runs = []
    for n in (64, 128, 256, 512):
        levels = int(np.log2(n // 64)) + 1
        p = dm.Params(shape=(n, n), window=(31, 31), levels=levels, descriptor=S3)
        D = dm.descriptor(torch.tensor(synthetic.checkerboard(n, a), dtype=torch.float32, device="cuda"), p)
        f = torch.empty(n, n, device="cuda")
        it, steps, secs = _exact_run(dm, torch, p, D, f, torch.zeros_like(f), torch.zeros_like(f), lr, cap)
        runs.append({"size": n, "levels": levels, "iterations_to_exact": it, "iterations_run": steps,
                     "seconds": round(secs, 3), "ms_per_iteration": round(1e3 * secs / max(steps, 1), 3)})
        print(json.dumps(runs[-1]), file=sys.stderr, flush=True)
    print(json.dumps({"metric": "checkerboards 64..512: iterations until the rounded field is exact", "unit": "iterations",
                      "config": {"descriptor": "S3 (Eq. s3)", "window": 31, "squares_px": a, "lr": lr,
                                 "levels": "down to 64x64", "test_every": 100, "max_iterations": cap},
                      "runs": runs}))
    return 0


def workload_config(args, wl, count, units, world) -> dict:
    """The workload, described the same way by both arms of the benchmark."""
    return {"workload": wl["desc"], "instances_per_gpu": count, "units_per_step": units,
            "l2": "flushed before every timed step (256 MB write)",
            "parallelism": "independent instances per GPU" if world > 1 else "single GPU"}


def make_instances(name: str, rank: int):
    """List of (shape, window, levels, target) for one rank."""
    wl = WORKLOADS[name]
    if wl.get("count"):
        return [(sh, w, wl["levels"], t) for sh, w, t in batch_instances(wl["count"], 4000 + 1000 * rank)]
    return [(wl["shape"], wl["window"], wl["levels"], make_target(name, rank))]


def make_target(name: str, seed_base: int) -> np.ndarray:
    if name == "mp3_512":
        return synthetic.multiphase_grf((512, 512), 12.0, (0.3, 0.3), 2000 + seed_base)
    if name == "grf512":
        return synthetic.target_large_2d(2000 + seed_base)
    if name == "grf128_3d":
        return synthetic.target_3d(128, 3000 + seed_base)
    return synthetic.target_small_2d(1000 + seed_base)


def units_per_step(shape, window, levels) -> int:
    kfull = int(np.prod([2 * p + 1 for p in window]))
    n = int(np.prod(shape))
    return sum((n >> (len(shape) * l)) * kfull for l in range(levels))


def level_sizes(shape, levels):
    return [int(np.prod([s >> l for s in shape])) for l in range(levels)]


# ----------------------------------------------------------------------------- clocks

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = os.path.join(tempfile.gettempdir(), "dmcr_clocks_%d.csv" % os.getpid())

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.f.close()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[5:9]):
                if val.lower() == "active":
                    reasons.add(nm)
        try:
            os.remove(self.path)
        except OSError:
            pass
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# ----------------------------------------------------------------------------- CPU oracle timing

def oracle_sample(shape, window, levels, target, field, budget_s: float, seed: int = 0):
    """Time the FP64 oracle on a bounded sample of one descriptor+gradient evaluation and
    extrapolate to voxel-shifts/s: forward on s half-window shifts of the finest level
    (N_1 pair evaluations each), VJP at q positions (2 K_half pair evaluations each)."""
    import oracle
    op = oracle.Params(ndim=len(shape), window=tuple(window), levels=levels)
    H = oracle.half_window(len(shape), window)
    K = H.shape[0]
    rng = np.random.default_rng(seed)
    M = np.asarray(field, dtype=np.float32).astype(np.float64)
    G = rng.standard_normal(K)
    N1 = M.size

    def run(s, q):
        idx = rng.choice(K, size=min(s, K), replace=False)
        t0 = time.perf_counter()
        oracle.sbar(M, H[idx])
        t1 = time.perf_counter()
        pos = rng.choice(N1, size=q, replace=False)
        oracle.level_vjp(M, op, G, pos)
        t2 = time.perf_counter()
        return (t1 - t0) / len(idx), (t2 - t1) / q

    tf, ta = run(8, 16)          # calibrate
    s = max(8, int(0.5 * budget_s / max(tf, 1e-9)))
    q = max(16, min(N1, int(0.5 * budget_s / max(ta, 1e-9))))
    tf, ta = run(s, q)
    sizes = level_sizes(shape, levels)
    t_full = sum(K * tf * (n / N1) + n * ta for n in sizes)
    units = units_per_step(shape, window, levels)
    return units / t_full, "%d forward shifts (of %d) on the %s level and the gradient at %d positions (of %d); " \
        "full step extrapolated over %d levels" % (s, K, "x".join(map(str, shape)), q, N1, levels)


def oracle_sample_mp(shape, window, levels, nph, field, budget_s: float, seed: int = 0):
    """Multi-phase form of ``oracle_sample``: forward on s half-window shifts of one phase
    pair of the finest level, the gradient of every phase at q finest positions (level 0),
    extrapolated to all nph^2 pairs and all levels."""
    import oracle
    op1 = oracle.Params(ndim=len(shape), window=tuple(window), levels=1)
    H = oracle.half_window(len(shape), window)
    K = H.shape[0]
    rng = np.random.default_rng(seed)
    F = np.asarray(field, dtype=np.float32).astype(np.float64)
    G = rng.standard_normal(nph * nph * K)
    N1 = F[0].size

    def run(s, q):
        idx = rng.choice(K, size=min(s, K), replace=False)
        t0 = time.perf_counter()
        oracle.cross_sbar(F[0], F[1], H[idx])
        t1 = time.perf_counter()
        oracle.multiphase_vjp_at(F, op1, G, rng.choice(N1, size=q, replace=False))
        t2 = time.perf_counter()
        return (t1 - t0) / len(idx), (t2 - t1) / q

    tf, ta = run(4, 2)           # calibrate
    s = max(4, int(0.5 * budget_s / max(tf, 1e-9)))
    q = max(2, min(N1, int(0.5 * budget_s / max(ta, 1e-9))))
    tf, ta = run(s, q)
    sizes = level_sizes(shape, levels)
    t_full = sum(nph * nph * K * tf * (n / N1) + n * ta for n in sizes)
    units = nph * nph * units_per_step(shape, window, levels)
    return units / t_full, "%d forward shifts (of %d) of one phase pair on the %s level and the gradient of all %d " \
        "phases at %d positions (of %d); full step extrapolated over %d phase pairs and %d levels" % (
            s, K, "x".join(map(str, shape)), nph, q, N1, nph * nph, levels)


PIPE_NAMES = ("rcp", "ex2", "tanh", "lg2", "ffma", "ffma2_lanes", "adjoint_pairs", "forward_pairs", "dfma")


def measure_pipe_rates() -> dict:
    """Measured throughput per SM per clock (libdmcr_pipes.so, csrc/pipes.cu): MUFU rcp /
    ex2 / tanh / lg2 operations, FFMA, FFMA2 lane operations, the pair rates of the
    adjoint's and the forward's per-pair arithmetic held in registers, and FP64 DFMA."""
    import ctypes
    from paper_2103_09686_gb300 import _build
    _build.build()
    lib = ctypes.CDLL(_build.PIPES_LIB)
    lib.dmcr_bench_pipe_rates.restype = ctypes.c_int
    r = (ctypes.c_double * len(PIPE_NAMES))()
    st = lib.dmcr_bench_pipe_rates(r)
    if st != 0:
        raise RuntimeError("pipe-rate probe failed with CUDA error %d" % st)
    return {k: float(r[i]) for i, k in enumerate(PIPE_NAMES)}


def cores_used() -> int:
    try:
        return int(os.environ.get("OMP_NUM_THREADS", "")) or os.cpu_count()
    except ValueError:
        return os.cpu_count()


# ----------------------------------------------------------------------------- main

def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=600)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="grf512", choices=sorted(WORKLOADS))
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-budget", type=float, default=16.0, help="seconds of oracle work for cpu_baseline")
    ap.add_argument("--serve", action="store_true", help="served vs plain reconstructions on a Poisson trace")
    ap.add_argument("--jobs", type=int, default=512, help="--serve: arrivals of the overload trace")
    ap.add_argument("--jobs2", type=int, default=128, help="--serve: arrivals of the trace at 80%% of capacity")
    ap.add_argument("--slots", type=int, default=64)
    ap.add_argument("--crossover", action="store_true", help="identity threshold: direct vs FFT over the window")
    ap.add_argument("--fft", action="store_true", help="FFT path roofline at 128^3 (identity threshold)")
    ap.add_argument("--pipes", action="store_true", help="measured MUFU / FMA rates per SM per clock")
    ap.add_argument("--tune", action="store_true", help="launch shapes from the autotuner (measured, cached)")
    ap.add_argument("--checkerboard", action="store_true", help="Sec. 4.1 checkerboard E1/E2 reconstructions")
    ap.add_argument("--s3", action="store_true", help="three-point descriptor steps at the paper's P = 31 configurations")
    ap.add_argument("--multigrid", action="store_true", help="Fig. reconstructionsmg: multigrid vs single-level vs coarse-to-fine")
    ap.add_argument("--c1", action="store_true",
                    help="the 64^2 +-16 workload as whole 200-iteration reconstructions: GPU vs the oracle on 1 "
                         "and all host cores")
    ap.add_argument("--checkerboard-sizes", action="store_true",
                    help="Fig. checerboardreconstructions: checkerboards of 64..512 with the multigrid scheme")
    args = ap.parse_args()
    if args.pipes:
        rates = measure_pipe_rates()
        print(json.dumps({"metric": "pipe rates", "unit": "per SM per clock", **rates}))
        return 0
    if args.serve:
        return main_serve(args)
    if args.crossover:
        return main_crossover(args)
    if args.fft:
        return main_fft(args)
    if args.checkerboard:
        return main_checkerboard(args)
    if args.s3:
        return main_s3(args)
    if args.multigrid:
        return main_multigrid(args)
    if args.checkerboard_sizes:
        return main_checkerboard_sizes(args)
    if args.c1:
        return main_c1(args)

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    wl = WORKLOADS[args.workload]
    nph = wl.get("phases", 1)
    insts = make_instances(args.workload, rank)
    units = nph * nph * sum(units_per_step(sh, w, lev) for sh, w, lev, _ in insts)
    big = max(insts, key=lambda x: int(np.prod(x[0])) * int(np.prod([2 * q + 1 for q in x[1]])))

    if args.impl == "reference":
        if rank != 0:
            return 0
        shape, window, levels, target = big
        field = synthetic.uniform_field(shape if nph == 1 else (nph,) + tuple(shape), seed=1)
        # about 150 s of oracle work for the whole run, however many steps it has
        per_step = max(0.1, min(8.0, 150.0 / max(1, args.steps + args.warmup)))
        vals, walls = [], []
        sample = ""
        for i in range(args.warmup + args.steps):
            t0 = time.perf_counter()
            if nph > 1:
                v, sample = oracle_sample_mp(shape, window, levels, nph, field, per_step, seed=i)
            else:
                v, sample = oracle_sample(shape, window, levels, target, field, per_step, seed=i)
            if i >= args.warmup:
                vals.append(v)
                walls.append(time.perf_counter() - t0)
        value = float(np.mean(vals))
        line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
                "steps": args.steps, "warmup": args.warmup,
                # wall time of one sampled step as run here; the time the oracle would need for
                # one whole step of the workload is extrapolated from the sample (next key)
                "ms_per_step": float(np.mean(walls)) * 1e3,
                "ms_per_full_step_extrapolated": units / value * 1e3,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
                "data": "synthetic", "config": workload_config(args, wl, len(insts), units, world),
                "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores_used(), "kind": "oracle",
                                 "sample": sample + "; value = sampled voxel-shifts / sampled oracle time "
                                           "(extrapolated rate, not a full step)"},
                "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(line))
        return 0

    import torch
    import paper_2103_09686_gb300 as dm
    dm.load()
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("gloo")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    pipes = measure_pipe_rates()      # the roofline's measured peaks (about 10 ms, before any timing)

    # inputs: this rank's own instances (weak scaling, no data-path collective)
    params = [dm.Params(shape=sh, window=w, levels=lev, phases=nph) for sh, w, lev, _ in insts]
    if args.tune:
        from paper_2103_09686_gb300 import tune
        params = [tune.tuned(p) for p in params]
    count = len(params)
    batched = count > 1
    opts = dm.ReconOpts(lr=1e-2)
    ws = dm.batch_workspace(params, dev) if batched else dm.workspace(params[0], dev)
    targets = [torch.tensor(t, dtype=torch.float32, device=dev) for _, _, _, t in insts]
    d_des = [torch.empty(dm.dmcr_descriptor_length(p), dtype=torch.float32, device=dev) for p in params]
    if batched:
        dm.dmcr_descriptor_batched(params, targets, d_des, ws)
    else:
        dm.dmcr_descriptor(params[0], targets[0], d_des[0], ws)
    fields0 = [torch.tensor(synthetic.uniform_field(sh if nph == 1 else (nph,) + tuple(sh), seed=7 + rank + 7919 * i),
                            dtype=torch.float32, device=dev)
               for i, (sh, _, _, _) in enumerate(insts)]
    fields = [f.clone() for f in fields0]
    ms = [torch.zeros_like(f) for f in fields]
    vs = [torch.zeros_like(f) for f in fields]
    loss = torch.empty(6 * count, dtype=torch.float32, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)     # > 129 MB L2
    steps = [0] * count
    stream = torch.cuda.current_stream()

    def one_step(tg, fl, st):
        if batched:
            return dm.dmcr_adam_step_batched(params, opts, tg, fl, ms, vs, st, loss, ws)
        return [dm.dmcr_adam_step(params[0], opts, tg[0], fl[0], ms[0], vs[0], st[0], loss, ws)]

    def barrier():
        if dist is not None:
            dist.barrier()

    for _ in range(args.warmup):
        steps = one_step(d_des, fields, steps)
    torch.cuda.synchronize()

    # ---- timed region: device-resident inputs, L2 flushed before every step; the library
    # replays its cached graph of the iteration (its per-kernel timers are off)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    sampler = ClockSampler(local)
    sampler.start()
    barrier()
    torch.cuda.synchronize()
    for k in range(args.steps):
        flush.zero_()
        ev[k][0].record(stream)
        steps = one_step(d_des, fields, steps)
        ev[k][1].record(stream)
    torch.cuda.synchronize()
    barrier()
    # ---- per-kernel durations for the roofline: the same steps with the library's event
    # timers on (direct launches, one event pair around each kernel)
    prof_steps = min(args.steps, 20)
    dm.dmcr_profile_reset()
    dm.dmcr_profile_enable(True)
    for k in range(prof_steps):
        flush.zero_()
        steps = one_step(d_des, fields, steps)
    torch.cuda.synchronize()
    dm.dmcr_profile_enable(False)
    clocks = sampler.stop()
    prof = dm.dmcr_profile_read()
    step_ms = [a.elapsed_time(b) for a, b in ev]
    total_s = sum(step_ms) / 1e3
    if dist is not None:
        t = torch.tensor([total_s], dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_s = float(t.item())
    value = units * args.steps * world / total_s
    loss_h = loss[:6].cpu().numpy().tolist()

    # ---- end to end through the C ABI with host buffers (pinned), copies inside the region
    h_fields = [f.cpu().pin_memory() for f in fields0]
    h_targets = [d.cpu().pin_memory() for d in d_des]
    h_loss = torch.empty(6 * count, dtype=torch.float32).pin_memory()
    e2e_steps = max(10, args.steps // 4)
    d_fields = [torch.empty_like(f) for f in fields]
    d_t = [torch.empty_like(d) for d in d_des]
    for m in ms:
        m.zero_()
    for v in vs:
        v.zero_()
    esteps = [0] * count
    # one untimed call with these buffers: the library captures its graph of the iteration here
    for a, b in zip(d_fields, h_fields):
        a.copy_(b, non_blocking=True)
    for a, b in zip(d_t, h_targets):
        a.copy_(b, non_blocking=True)
    one_step(d_t, d_fields, esteps)
    for m in ms:
        m.zero_()
    for v in vs:
        v.zero_()
    barrier()
    torch.cuda.synchronize()
    e2e_s = 0.0
    for k in range(e2e_steps):
        # as in the timed loop, L2 is flushed between steps (outside the timed windows): no
        # step finds its inputs L2-resident; each window runs from the host's first copy to
        # the loss back in host memory
        flush.zero_()
        torch.cuda.current_stream().synchronize()
        t0 = time.perf_counter()
        for a, b in zip(d_fields, h_fields):
            a.copy_(b, non_blocking=True)
        for a, b in zip(d_t, h_targets):
            a.copy_(b, non_blocking=True)
        esteps = one_step(d_t, d_fields, esteps)
        h_loss.copy_(loss, non_blocking=True)
        torch.cuda.current_stream().synchronize()
        e2e_s += time.perf_counter() - t0
    barrier()
    if dist is not None:
        t = torch.tensor([e2e_s], dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        e2e_s = float(t.item())
    e2e_value = units * e2e_steps * world / e2e_s
    h2d = sum(h.numel() * 4 for h in h_fields) + sum(h.numel() * 4 for h in h_targets)
    d2h = h_loss.numel() * 4

    # ---- roofline of the dominant kernel (largest summed duration in the timed region);
    # the correlation kernels are one fused launch over all levels (and instances)
    name, (kms, kcnt) = max(prof.items(), key=lambda kv: kv[1][0])
    pairs_adj = pairs_fwd = 0
    for sh, w, lev, _ in insts:
        kfull = int(np.prod([2 * q + 1 for q in w]))
        nsum = nph * nph * sum(level_sizes(sh, lev))
        pairs_adj += nsum * kfull
        pairs_fwd += nsum * ((kfull + 1) // 2)
    pairs = pairs_adj if name.startswith("corr_adj") else (pairs_fwd if name.startswith("corr_fwd") else None)
    # separable instances evaluate no pairs (their gated correlation launches find nothing to do)
    separable = any(k.startswith("sep_") for k in prof)
    if separable:
        pairs = None
    sm_count = torch.cuda.get_device_properties(dev).multi_processor_count
    max_mhz = clocks.get("sm_max_mhz") or 2070.0
    avg_ms = kms / max(kcnt, 1)
    roofline = None
    if pairs is not None:
        kind = "corr_adj" if name.startswith("corr_adj") else "corr_fwd"
        t = avg_ms / 1e3
        clk = max_mhz * 1e6
        # peaks from the pipe-rate probe run on this GPU (independent FFMA2 streams, MUFU rcp,
        # each kernel's instruction mix in registers), per SM per clock x SMs x max SM clock
        peak = sm_count * pipes["ffma2_lanes"] * clk / 1e12                    # T lane-op/s
        achieved = pairs * LANE_OPS_PER_PAIR[kind] / t / 1e12
        mufu_peak = sm_count * pipes["rcp"] * clk / 1e12                       # T rcp/s
        mufu = pairs * RCP_PER_PAIR[kind] / t / 1e12
        mix_peak = sm_count * pipes[MIX_KEY[kind]] * clk                       # pairs/s
        nominal = sm_count * FP32_LANES_NOMINAL * clk / 1e12
        roofline = {"bound": "alu", "kernel": name, "achieved": achieved, "peak": peak, "unit": "Tlane-op/s",
                    "frac": achieved / peak, "traffic": NCU_TRAFFIC_BYTES.get((args.workload, kind)),
                    "peak_basis": "measured FP32 pipe: %d SMs x %.1f FFMA2 lane-ops/clk (probe, independent streams) "
                                  "x %.0f MHz (max SM clock); achieved = algorithmic pairs x %.4g implemented FP32 "
                                  "lane-ops/pair / launch time" % (sm_count, pipes["ffma2_lanes"], max_mhz,
                                                                   LANE_OPS_PER_PAIR[kind]),
                    "nominal": {"peak": nominal, "frac": achieved / nominal,
                                "basis": "%d FP32 lanes/clk/SM by unit count" % FP32_LANES_NOMINAL},
                    "algorithmic": {"fp32_ops_per_pair": ALGORITHMIC_FP32_OPS_PER_PAIR,
                                    "achieved": pairs * ALGORITHMIC_FP32_OPS_PER_PAIR / t / 1e12,
                                    "frac": pairs * ALGORITHMIC_FP32_OPS_PER_PAIR / t / 1e12 / peak},
                    "mufu": {"achieved": mufu, "peak": mufu_peak, "unit": "Trcp/s", "frac": mufu / mufu_peak,
                             "rcp_per_pair": RCP_PER_PAIR[kind], "basis": "measured MUFU rcp %.2f/clk/SM" % pipes["rcp"]},
                    "mix_ceiling": {"pairs_per_s": mix_peak, "frac": pairs / t / mix_peak,
                                    "basis": "the kernel's per-pair instruction mix in registers, measured %.2f "
                                             "pairs/clk/SM" % pipes[MIX_KEY[kind]]},
                    "binding_frac": max(achieved / peak, mufu / mufu_peak),
                    "pairs_per_launch": pairs, "pairs_per_s": pairs / t,
                    "avg_launch_ms": avg_ms, "launches": kcnt}
    elif separable:
        # the step against what no method avoids: a transform there and back for the correlation
        # of each ordered phase pair and its gradient the same again, 5 N log2 N operations each
        flops = sum(nph * nph * 4 * 5.0 * n * np.log2(n) for sh, _, lev, _ in insts for n in level_sizes(sh, lev))
        peak = sm_count * pipes["ffma2_lanes"] * 2 * max_mhz * 1e6 / 1e12
        achieved = flops / (total_s / args.steps) / 1e12
        step_ms = total_s / args.steps * 1e3
        roofline = {"bound": "alu", "kernel": "whole step", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                    "frac": achieved / peak, "traffic": None,
                    "peak_basis": "measured FP32 pipe (FFMA2 probe) at the max SM clock; achieved = transform "
                                  "operations of the exact correlation and its gradient / step time (the separable "
                                  "path runs about a dozen such transforms, one per pair of features)",
                    "avg_launch_ms": step_ms, "launches": args.steps,
                    "slowest_kernel": {"kernel": name, "avg_launch_ms": avg_ms, "launches": kcnt}}
    # kernels of this library per step (the profiled pass launches the kernels of a graph replay
    # directly), times steps
    launches = int(round(sum(c for _, c in prof.values()) / max(prof_steps, 1) * args.steps))

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        shape, window, levels, target = big
        if nph > 1:
            v_cpu, sample = oracle_sample_mp(shape, window, levels, nph,
                                             synthetic.uniform_field((nph,) + tuple(shape), seed=7), args.cpu_budget)
        else:
            v_cpu, sample = oracle_sample(shape, window, levels, target, synthetic.uniform_field(shape, seed=7),
                                          args.cpu_budget)
        cpu = {"value": v_cpu, "unit": UNIT, "cores": cores_used(), "kind": "oracle", "sample": sample}

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": total_s * 1e3 / args.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
                "config": workload_config(args, wl, count, units, world),
                "launch_shapes": "autotuned %s" % sorted({tuple(p.tune) for p in params})
                if args.tune else "built-in plan",
                "roofline": roofline, "cpu_baseline": cpu,
                "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
                        "d2h_bytes_per_step": int(d2h), "steps": e2e_steps,
                        "l2": "flushed before every step, outside the per-step wall-clock windows (as in the timed loop)"},
                "gpu_launches": launches, "clocks": clocks,
                "kernels": {k: {"ms": round(t, 4), "launches": c} for k, (t, c) in sorted(prof.items())},
                "kernels_basis": "event-timed direct launches over %d further steps (timers on)" % prof_steps,
                "profiled_ms_per_step": sum(t for t, _ in prof.values()) / max(prof_steps, 1),
                "final_loss": loss_h}
        print(json.dumps(line))
    if dist is not None:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
