"""Benchmark: unbounded LGF Poisson solve throughput on one GB300 (or N replicas).

Workload (default): the 128^3 vector streamfunction solve a = -L^{-1} w of a
tilted Gaussian-core vortex ring (R = 32, sigma = 3 cells, circulation 1),
16^3 blocks, sources on the blocks where |w| > 1e-14 max, results on all 512
blocks, FP32 data, seeded synthetic input.  One step = one lgf_conv_execute
(all three components, one stream each, replayed as a CUDA graph).  Points =
target points x components.

Timing: W warm-up steps, then exactly K steps, each bracketed by CUDA events
on the launching stream; a 256 MiB buffer (> the 129 MB L2) is rewritten
between steps, outside the events.  Barrier + synchronize on both sides; the
max over ranks is reported.  Under torchrun every rank runs its own replica of
the solve (weak scaling, no data-path collective).

Extra keys: roofline (dominant kernel: the path's algorithmic 8 B per target
point and component of one launch / its mean event time, against the measured
HBM copy bandwidth; the whole step on the same rule), compute_roofline (the
dominant pass's algorithmic flops against the FP32 FMA rate measured in the
run by lgf_measure_peak), cpu_baseline (the FP64
oracle's direct sum on a bounded sample of target points, host cores),
e2e (the same solve through lgf_conv_execute_host with pinned host buffers,
copies included), gpu_launches, clocks (nvidia-smi sampled during the run).

--impl reference runs the FP64 CPU oracle (direct summation, the program the
GPU path is checked against) on the same workload, each step a bounded sample
of target points.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "Mpoints/s per unbounded LGF Poisson solve at 1e-6 rel err; % of roofline"
UNIT = "Mpoints/s"
B = 16


def workload():
    from paper_1601_00035_gb300 import inputs
    w, axis = inputs.ring_128()
    src_c = inputs.active_blocks(w, B, 1e-14)
    dst_c = inputs.block_grid(w.shape[1:], B)
    f = inputs.to_blocks(w, B, src_c)
    cfg = {"workload": "vortex-ring streamfunction a = -L^-1 w, 128^3 box, 3 components, 16^3 blocks",
           "box": [128, 128, 128], "block": B, "components": 3, "src_blocks": int(len(src_c)),
           "dst_blocks": int(len(dst_c)), "ring": {"R": 32, "sigma": 3, "gamma": 1, "axis": [round(float(a), 4) for a in axis]},
           "source_threshold": "blocks with |w| > 1e-14 max"}
    return f, src_c, dst_c, cfg


def max_over_ranks(x: float, device=None) -> float:
    """Largest value of x over the ranks of the default process group (x itself
    without one); the whole-job time is the slowest rank's."""
    import torch
    import torch.distributed as tdist
    if not (tdist.is_available() and tdist.is_initialized()) or tdist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    tdist.all_reduce(t, op=tdist.ReduceOp.MAX)
    return float(t.item())


def job_rate(units_per_rank_step: float, steps: int, world: int, seconds: float) -> float:
    """Whole-job throughput in millions of units per second: every rank
    processes the same per-step work (replicas, weak scaling) and the job ends
    with the slowest rank."""
    return units_per_rank_step * steps * world / seconds / 1e6


def rank_info():
    r = int(os.environ.get("RANK", "0"))
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    lr = int(os.environ.get("LOCAL_RANK", "0"))
    return r, ws, lr


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            p = json.load(fh)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def clock_sampler(gpu_index: int):
    q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
    try:
        return subprocess.Popen(["nvidia-smi", "-i", str(gpu_index), "--query-gpu=" + q, "--format=csv,noheader,nounits",
                                 "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
    except Exception:
        return None


def clock_summary(proc):
    if proc is None:
        return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
    proc.terminate()
    try:
        out, _ = proc.communicate(timeout=5)
    except Exception:
        proc.kill()
        out = ""
    sms, mx, reasons = [], None, set()
    names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
    for line in out.strip().splitlines():
        f = [x.strip() for x in line.split(",")]
        if len(f) < 9:
            continue
        try:
            sms.append(float(f[1]))
            mx = float(f[2])
        except ValueError:
            continue
        for n, v in zip(names, f[5:9]):
            if v.lower().startswith("active"):
                reasons.add(n)
    return {"sm_mhz": statistics.median(sms) if sms else None, "sm_max_mhz": mx, "samples": len(sms),
            "reasons": sorted(reasons)}


def pass_bytes(plan_geom):
    """Bytes each FFT pass must read and write (its own input and output arrays),
    from the plan geometry; complex FP32 = 8 B, real FP32 = 4 B."""
    g = plan_geom
    nc, KX = g["ncomp"], g["N"][0] // 2 + 1
    Es, Et, N = g["Es"], g["Et"], g["N"]
    X1 = nc * Es[2] * Es[1] * KX * 8
    X2 = nc * Es[2] * N[1] * KX * 8
    X3 = nc * Et[2] * N[1] * KX * 8
    X4 = nc * Et[2] * Et[1] * KX * 8
    Kh = (N[0] // 2 + 1) * (N[1] // 2 + 1) * (N[2] // 2 + 1) * 4
    Kt = (N[0] // 2 + 1) * N[1] * (N[2] // 2 + 1) * 4  # three-pass form: all of y
    src = g["nsrc"] * nc * B ** 3 * 4
    dst = g["ndst"] * nc * B ** 3 * 4
    return {"x_fwd_gather_r2c": src + X1, "y_fwd": X1 + X2, "z_fwd_mul_inv": X2 + Kh + X3, "y_inv": X3 + X4,
            "yz_conv": X1 + Kt + X4, "x_inv_c2r_scatter": X4 + dst}


def geometry(src_c, dst_c, ncomp, lengths):
    """Boxes, block counts and the FFT lengths (x, y, z) that the plan runs on."""
    s, t = np.asarray(src_c), np.asarray(dst_c)
    Es = [int((s[:, a].max() - s[:, a].min() + 1) * B) for a in range(3)]
    Et = [int((t[:, a].max() - t[:, a].min() + 1) * B) for a in range(3)]
    return {"Es": Es, "Et": Et, "N": list(lengths), "ncomp": ncomp, "nsrc": len(s), "ndst": len(t)}


def pass_flops(plan_geom):
    """Algorithmic flops of each FFT pass of one launch: 5 n log2 n per complex
    n-point transform (a real n-point transform counts as half of one), two
    transforms per z line plus 2 flops per point of the real spectral multiply."""
    g = plan_geom
    nc, N, Es, Et = g["ncomp"], g["N"], g["Es"], g["Et"]
    KX = N[0] // 2 + 1

    def c(n):
        return 5.0 * n * math.log2(n)
    y_fwd, y_inv = nc * Es[2] * KX * c(N[1]), nc * Et[2] * KX * c(N[1])
    z = nc * N[1] * KX * (2 * c(N[2]) + 2 * N[2])
    return {"x_fwd_gather_r2c": nc * Es[2] * Es[1] * c(N[0]) / 2,
            "y_fwd": y_fwd, "z_fwd_mul_inv": z, "y_inv": y_inv, "yz_conv": y_fwd + z + y_inv,
            "x_inv_c2r_scatter": nc * Et[2] * Et[1] * c(N[0]) / 2}


def oracle_sampler(f, src_c, rng_seed: int = 11):
    """The FP64 direct sum (the oracle, as it stands) prepared on the workload's
    sources; returns (run, ncomp, threads), run(n) timing n random target
    points per component in seconds."""
    import oracle as O
    from paper_1601_00035_gb300 import inputs
    cube = O.lgf_cube(127)
    pts_src = inputs.block_points(src_c, B)
    comps = []
    for c in range(f.shape[1]):
        v = f[:, c].reshape(-1).astype(np.float64)
        nz = v != 0
        comps.append((pts_src[nz], v[nz]))
    rng = np.random.default_rng(rng_seed)

    def run(n):
        tgt = rng.integers(0, 128, size=(n, 3)).astype(np.int32)
        t0 = time.perf_counter()
        for sp, sv in comps:
            O.direct_conv(cube, sp, -sv, tgt)
        return time.perf_counter() - t0

    return run, len(comps), O.num_threads()


def calibrate(run, target_seconds: float) -> int:
    """Sample size whose run takes about target_seconds: grow the sample until
    the fixed cost of a call is amortised, then scale."""
    n, t = 24, run(24)
    enough = min(target_seconds / 2, max(target_seconds / 16, 0.25))
    while t < enough and n < 1 << 22:
        n *= 4
        t = run(n)
    return max(24, int(n * target_seconds / max(t, 1e-3)))


def cpu_oracle_rate(f, src_c, target_seconds: float, rng_seed: int = 11):
    """Mpoints/s of the oracle on one bounded sample of about target_seconds;
    returns (Mpoints/s, points, seconds, threads)."""
    run, nc, thr = oracle_sampler(f, src_c, rng_seed)
    n = calibrate(run, target_seconds)
    dt = run(n)
    return n * nc / dt / 1e6, n * nc, dt, thr


def cpu_fft_rate(f, src_c, dst_c, u_gpu, reps: int = 2):
    """The same solve on the host by the oracle's FP64 zero-padded FFT convolution
    (oracle.fft_conv: scipy.fft on every core, G from the oracle's table), the
    fast-CPU reference point beside the direct sum.  Returns (Mpoints/s, seconds
    per solve, threads, relative L2 difference to the GPU result at 4096 sampled
    targets)."""
    import oracle as O
    from paper_1601_00035_gb300 import inputs
    nc = f.shape[1]
    s, t = np.asarray(src_c), np.asarray(dst_c)
    s0, s1 = s.min(0) * B, (s.max(0) + 1) * B
    t0, t1 = t.min(0) * B, (t.max(0) + 1) * B
    workers = os.cpu_count() or 1
    times = []
    for _ in range(reps):
        a = time.perf_counter()
        F = np.zeros((nc, *(s1 - s0)[::-1]))
        for b, (bx, by, bz) in enumerate(s * B - s0):
            F[:, bz:bz + B, by:by + B, bx:bx + B] = f[b]
        U = -O.fft_conv(F, s0, t0, tuple((t1 - t0)[::-1]), workers=workers)
        times.append(time.perf_counter() - a)
    tgt = inputs.block_points(dst_c, B)
    sel = np.random.default_rng(5).choice(len(tgt), 4096, replace=False)
    tx, ty, tz = [tgt[sel, a] - t0[a] for a in range(3)]
    diff = 0.0
    for c in range(nc):
        ref = U[c][tz, ty, tx]
        got = u_gpu[(sel // B ** 3), c].reshape(-1, B ** 3)[np.arange(len(sel)), sel % B ** 3]
        diff = max(diff, float(np.linalg.norm(got - ref) / np.linalg.norm(ref)))
    dt = min(times)
    return len(dst_c) * B ** 3 * nc / dt / 1e6, dt, workers, diff


def bench_reference(args):
    r, ws, lr = rank_info()
    if r != 0:
        return 0
    f, src_c, dst_c, cfg = workload()
    # each step a bounded sample; the whole run stays within a few minutes
    per_step = float(os.environ.get("LGF_REF_STEP_SECONDS", "2.0"))
    per_step = min(per_step, max(0.25, 150.0 / (args.steps + args.warmup)))
    run, nc, thr = oracle_sampler(f, src_c, rng_seed=100)
    n = calibrate(run, per_step)
    times = []
    for i in range(args.warmup + args.steps):
        dt = run(n)
        if i >= args.warmup:
            times.append(dt)
    total = sum(times)
    value = n * nc * len(times) / total / 1e6
    line = {"metric": METRIC, "value": value, "unit": UNIT, "impl": "reference", "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * total / len(times), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": cfg,
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": thr, "kind": "oracle",
                             "sample": "FP64 direct sum at %d random target points x %d components per step "
                                       "(~%.2f s of host work each)" % (n, nc, per_step)},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def bench_gpu(args):
    import torch
    r, ws, lr = rank_info()
    dist = ws > 1
    if dist:
        import torch.distributed as tdist
        torch.cuda.set_device(lr)
        tdist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    from paper_1601_00035_gb300 import build as libbuild
    libbuild.build()
    from paper_1601_00035_gb300 import lgf

    f, src_c, dst_c, cfg = workload()
    K = lgf.required_max_offset(src_c, dst_c, B)
    table = lgf.Table(lgf.LAPLACE7, max_offset=K)
    # the library runs the three components in each launch of its three passes (or, five passes, on
    # three streams); the launch sequence is captured in a CUDA graph on first use
    plan = lgf.Plan(table, [lgf.Solve(B, 3, src_c, dst_c, scale=-1.0)], use_graph=True, method=lgf.METHOD_AUTOTUNE)
    chosen, auto_wb, auto_split = plan.method()
    passes, lengths = plan.lengths()
    stream = torch.cuda.current_stream()
    d_src = torch.from_numpy(f).cuda()
    d_dst = torch.zeros((len(dst_c), 3, B, B, B), device="cuda")
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    pts_per_step = len(dst_c) * B ** 3 * 3

    # measured arithmetic peaks (compute roofline of the FFT passes), before the timed region
    peaks_tf = {k: round(lgf.measure_peak(v, 200.0), 2) for k, v in
                (("fp32_fma", lgf.PEAK_FP32), ("fp32x2_fma", lgf.PEAK_FP32X2), ("fp64_fma", lgf.PEAK_FP64))}
    sampler = clock_sampler(torch.cuda.current_device()) if r == 0 else None
    time.sleep(0.5)
    for _ in range(args.warmup):
        plan.execute([d_src], [d_dst])
        flush.fill_(1.0)
    torch.cuda.synchronize()
    if dist:
        tdist.barrier()
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    wall0 = time.perf_counter()
    for i in range(args.steps):
        flush.fill_(float(i))
        ev[i][0].record(stream)
        plan.execute([d_src], [d_dst])
        ev[i][1].record(stream)
    torch.cuda.synchronize()
    wall = time.perf_counter() - wall0
    step_ms = [a.elapsed_time(b) for a, b in ev]
    dev_ms = sum(step_ms)
    # per-pass durations: the same K steps again with an event pair around every
    # pass (the library's profiling mode).  The events serialise the passes, which
    # otherwise overlap at their boundaries (programmatic dependent launch), so
    # this replay runs a little longer than the timed region above.
    plan.set_profiling(2)
    for i in range(args.steps):
        flush.fill_(float(i))
        plan.execute([d_src], [d_dst])
    torch.cuda.synchronize()
    plan.set_profiling(0)
    kt = plan.kernel_times()
    if dist:
        dev_ms = max_over_ranks(dev_ms, device="cuda")
        tdist.barrier()
    torch.cuda.synchronize()
    clocks = clock_summary(sampler) if r == 0 else None

    # the plain form for comparison (outside the timed region): one component per
    # solve, the three solves one after another on one stream, no graph
    plain = lgf.Plan(table, [lgf.Solve(B, 1, src_c, dst_c, scale=-1.0)])
    srcs1 = [d_src[:, q:q + 1].contiguous() for q in range(3)]
    dsts1 = [torch.zeros((len(dst_c), 1, B, B, B), device="cuda") for _ in range(3)]

    def run_plain():
        for a, b in zip(srcs1, dsts1):
            plain.execute([a], [b])
    plain_ms = _timed_ms(torch, run_plain)

    # e2e: host (pinned) buffers through lgf_conv_execute_host, copies included
    h_src = torch.from_numpy(f).pin_memory()
    h_dst = torch.empty((len(dst_c), 3, B, B, B), dtype=torch.float32).pin_memory()
    e2e_steps = max(3, min(args.steps, 50))
    for _ in range(2):
        plan.execute_host([h_src], [h_dst])
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        plan.execute_host([h_src], [h_dst])
    e2e_s = time.perf_counter() - t0
    if dist:
        e2e_s = max_over_ranks(e2e_s, device="cuda")

    if r != 0:
        if dist:
            tdist.destroy_process_group()
        return 0

    value = job_rate(pts_per_step, args.steps, ws, dev_ms / 1e3)
    e2e_value = job_rate(pts_per_step, e2e_steps, ws, e2e_s)
    # roofline of the dominant kernel, on the algorithmic bytes of the path: 8 B per target
    # point (4 B FP32 source in, 4 B result out); one launch of a pass is all three components
    # in the three-pass form, one component in the five-pass form
    per = 3 if passes == 3 else 1
    g1 = geometry(src_c, dst_c, per, lengths)
    # (the autotuner may have chosen the split solve: no per-pass workspace or flop model)
    pb, pf = (pass_bytes(g1), pass_flops(g1)) if passes else ({}, {})
    dom = max(kt, key=lambda k: kt[k][1])
    launches, tot_ms = kt[dom]
    per_launch_ms = tot_ms / launches
    hbm, src_kind = peaks()
    alg_bytes = 8 * per * len(dst_c) * B ** 3
    achieved = alg_bytes / (per_launch_ms / 1e3) / 1e9
    if dom not in pb:
        pb[dom], pf[dom] = 0, 0.0
    step_gbs = 8 * pts_per_step / (dev_ms / args.steps / 1e3) / 1e9
    roof = {"bound": "hbm", "kernel": dom, "achieved": round(achieved, 1), "peak": hbm, "unit": "GB/s",
            "frac": round(achieved / hbm, 4), "traffic": None,
            "algorithmic_bytes_per_launch": alg_bytes, "mean_launch_ms": round(per_launch_ms, 5),
            "bytes_rule": "8 B per target point and component (FP32 source read + result write), %d component(s) "
                          "per launch" % per,
            "step": {"achieved": round(step_gbs, 1), "frac": round(step_gbs / hbm, 4),
                     "rule": "8 B per target point and component over the whole timed step"},
            "pass_workspace": {"bytes_per_launch": pb[dom],
                               "achieved": round(pb[dom] / (per_launch_ms / 1e3) / 1e9, 1),
                               "frac": round(pb[dom] / (per_launch_ms / 1e3) / 1e9 / hbm, 4),
                               "rule": "the pass's own input and output arrays (complex FP32 workspaces, "
                                       "kernel spectrum): bytes of this algorithm, not of the path"},
            "traffic_note": "DRAM bytes per launch are counted by ncu, not in this run",
            "launch_timing": "CUDA events around each launch (one pass) in K profiled steps after the timed ones",
            "peak_source": src_kind + " (MEASURED_PEAKS.json hbm_gbs)" if src_kind == "measured" else src_kind}
    comp_tf = pf[dom] / (per_launch_ms / 1e3) / 1e12
    compute = {"bound": "fp32", "kernel": dom, "achieved": round(comp_tf, 2), "peak": peaks_tf["fp32_fma"],
               "unit": "TFLOP/s", "frac": round(comp_tf / peaks_tf["fp32_fma"], 4),
               "flops_per_launch": pf[dom],
               "flop_rule": "5 n log2 n per complex n-point transform (real: half), 2 per spectral-multiply point",
               "peaks_measured_tflops": peaks_tf,
               "peak_source": "lgf_measure_peak: FMA chains on every SM, CUDA events, measured in this run"}
    shares = {k: {"launches": v[0], "ms": round(v[1], 4), "share": round(v[1] / sum(x[1] for x in kt.values()), 4),
                  "workspace_gbs": round(pb.get(k, 0) * v[0] / (v[1] / 1e3) / 1e9, 1),
                  "tflops": round(pf.get(k, 0.0) * v[0] / (v[1] / 1e3) / 1e12, 2)} for k, v in kt.items()}
    # CPU baseline: oracle on a bounded sample (rank 0, N=1 only)
    cpu = cpu_fft = None
    if ws == 1 and not args.no_cpu_baseline:
        rate, pts, dt, thr = cpu_oracle_rate(f, src_c, args.cpu_seconds)
        cpu = {"value": rate, "unit": UNIT, "cores": thr, "kind": "oracle",
               "sample": "FP64 direct sum (oracle) at %d random target points x 3 components, %.1f s" % (pts // 3, dt)}
        frate, fdt, fthr, fdiff = cpu_fft_rate(f, src_c, dst_c, d_dst.cpu().numpy())
        cpu_fft = {"value": round(frate, 2), "unit": UNIT, "cores": fthr,
                   "kind": "FP64 zero-padded FFT convolution on the host (oracle.fft_conv: scipy.fft, G from the "
                           "oracle's table)",
                   "sample": "the full solve, best of 2: %.2f s" % fdt, "rel_l2_vs_gpu": fdiff}
    cfg = dict(cfg)
    cfg.update({"method": {"chosen": ["whole-box FFT convolution", "block-sparse split solve"][chosen],
                           "autotune_ms": {"whole_box": round(auto_wb, 4), "split": round(auto_split, 4)},
                           "rule": "lgf_conv_plan method 2: both planned, one timed execution each, the faster kept"},
                "fft_grid": lengths, "execution": "%s, launch sequence replayed as a CUDA graph" %
                ("three passes, all components per launch" if per == 3 else "one stream per component"),
                "plain_ms": round(plain_ms, 4), "batched_over_plain": round(plain_ms / (dev_ms / args.steps), 3),
                "plain": "one component per solve, three solves one after another on one stream, no graph",
                "l2": "256 MiB buffer rewritten between timed steps (outside the events)",
                "precision": "FP32 data and FFTs; FP64 LGF table and kernel spectrum",
                "parity": "rel L2 <= 1e-6 vs FP64 direct sum (tests/test_gpu_poisson.py)"})
    line = {"metric": METRIC, "value": round(value, 1), "unit": UNIT, "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": round(dev_ms / args.steps, 5), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic", "config": cfg,
            "roofline": roof, "compute_roofline": compute, "kernels": shares, "cpu_baseline": cpu, "cpu_fft_baseline": cpu_fft,
            "e2e": {"value": round(e2e_value, 1), "unit": UNIT, "h2d_bytes_per_step": int(f.nbytes),
                    "d2h_bytes_per_step": int(h_dst.numel() * 4)},
            "gpu_launches": int(sum(v[0] for v in kt.values())), "clocks": clocks,
            "wall_s_timed_region": round(wall, 4)}
    print(json.dumps(line))
    if dist:
        tdist.destroy_process_group()
    return 0


# ---------------------------------------------------------------------------
# other workloads (not the headline metric): each prints one JSON line with its
# own metric; device time with CUDA events, L2 flushed between steps.
# ---------------------------------------------------------------------------
def _dilate(blocks):
    s = set(map(tuple, np.asarray(blocks).tolist()))
    out = set()
    for (x, y, z) in s:
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    out.add((x + dx, y + dy, z + dz))
    return np.array(sorted(out), dtype=np.int32)


def aux_workload(name, lgf, torch):
    """Returns (step_fn, plans, points_per_step, config, graph_note)."""
    from paper_1601_00035_gb300 import inputs
    if name == "blobs32":
        f = inputs.gaussian_blobs(32)
        c = inputs.block_grid(f.shape, B)
        t = lgf.Table(lgf.LAPLACE7, max_offset=lgf.required_max_offset(c, c, B))
        p = lgf.Plan(t, [lgf.Solve(B, 1, c, c)])
        src = torch.from_numpy(inputs.to_blocks(f, B, c)).cuda()
        dst = torch.zeros_like(src)
        return (lambda: p.execute([src], [dst])), [p], 32 ** 3, {
            "workload": "scalar Poisson, 32^3 box, 3 Gaussian blobs, 16^3 blocks"}, [t]
    if name == "blobs32_f64":
        # the same solve with FP64 data, transforms and spectrum (plan precision 1)
        f = inputs.gaussian_blobs(32)
        c = inputs.block_grid(f.shape, B)
        t = lgf.Table(lgf.LAPLACE7, max_offset=lgf.required_max_offset(c, c, B))
        p = lgf.Plan(t, [lgf.Solve(B, 1, c, c)], precision=1)
        src = torch.from_numpy(inputs.to_blocks(f, B, c, dtype=np.float64)).cuda()
        dst = torch.zeros_like(src)
        return (lambda: p.execute_f64([src], [dst])), [p], 32 ** 3, {
            "workload": "scalar Poisson in FP64, 32^3 box, 3 Gaussian blobs, 16^3 blocks"}, [t]
    if name == "if128":
        u = inputs.two_ring_velocity()
        c = inputs.block_grid(u.shape[1:], B)
        x = torch.from_numpy(inputs.to_blocks(u, B, c)).cuda()
        ys = [torch.zeros_like(x) for _ in range(3)]
        tabs = [lgf.Table(lgf.IFACTOR, alpha=a) for a in (0.05, 0.2, 1.0)]
        plans = [lgf.Plan(tb, [lgf.Solve(B, 3, c, None)]) for tb in tabs]
        f = inputs.gaussian_blobs(32)
        cb = inputs.block_grid(f.shape, B)
        tp = lgf.Table(lgf.LAPLACE7, max_offset=lgf.required_max_offset(cb, cb, B))
        pp = lgf.Plan(tp, [lgf.Solve(B, 1, cb, cb)])
        fs = torch.from_numpy(inputs.to_blocks(f, B, cb)).cuda()
        fd = torch.zeros_like(fs)

        def step():
            for pl, y in zip(plans, ys):
                pl.ifactor(x, y)
            pp.execute([fs], [fd])
        # the plain form for comparison: one component per application, separate
        # launches on one stream, no graph
        plans1 = [lgf.Plan(tb, [lgf.Solve(B, 1, c, None)]) for tb in tabs]
        x1 = [x[:, q:q + 1].contiguous() for q in range(3)]
        y1 = [torch.zeros_like(x1[0]) for _ in range(3)]

        def run_plain():
            for pl in plans1:
                for q in range(3):
                    pl.ifactor(x1[q], y1[q])
            pp.execute([fs], [fd])
        plain_ms = _timed_ms(torch, run_plain)
        g = torch.cuda.CUDAGraph()
        step()
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            step()
        batched_ms = _timed_ms(torch, g.replay)
        return step, plans + [pp], 3 * x.numel() + 32 ** 3, {
            "workload": "integrating factor on a 3 x 128^3 two-ring velocity, alpha in {0.05, 0.2, 1.0} "
                        "(R = 7, 9, 15), plus the 32^3 Poisson solve, one captured graph per step",
            "plain_ms": round(plain_ms, 4), "batched_ms": round(batched_ms, 4),
            "batched_over_plain": round(plain_ms / batched_ms, 3),
            "plain": "one component per integrating-factor application (9 applications) and the Poisson "
                     "solve, separate launches on one stream, no graph"}, tabs + [tp]
    if name in ("rk256", "rk256_b", "rk256_c", "rk256_refresh", "rk256_vort"):
        n, R0c, dcells = 256, 50.0, 10.0
        dx = 1.0 / R0c                      # R0 = 1, Gamma = 1
        dt, re = 0.01721, 500.0             # Sec. 6.4: dt Gamma/R0^2 = 0.01721, Re = 500
        uinf = (0.0, 0.0, -0.18686)
        axis = inputs.random_axis_tilted(inputs.rng_for(4))
        w = inputs.vortex_ring_edges(n, R0c, dcells, axis) / dx ** 2   # physical vorticity
        supp = inputs.active_blocks(w, B, 1e-6)
        scheme = {"rk256": 0, "rk256_b": 1, "rk256_c": 2, "rk256_refresh": 0, "rk256_vort": 0}[name]
        rk = lgf.RKPlan(B, supp, dx, dt, re, scheme=scheme, use_graph=True)
        xs = rk.blocks(0)
        # initial velocity by the method itself: a = -L^-1 w (vector, D_supp -> D_xsoln), u = C^T a
        K = lgf.required_max_offset(supp, xs, B)
        t = lgf.Table(lgf.LAPLACE7, max_offset=K)
        pv = lgf.Plan(t, [lgf.Solve(B, 3, supp, xs, dx=dx, scale=-1.0)])
        ws = torch.from_numpy(inputs.to_blocks(w, B, supp)).cuda()
        a = torch.zeros((len(xs), 3, B, B, B), device="cuda")
        pv.execute([ws], [a])
        u0 = torch.zeros_like(a)
        rk.op(lgf.OP_CURL_T, a, u0)
        u1 = torch.zeros_like(u0)
        if name == "rk256_vort":
            # the vorticity formulation of Sec. 4.1: a vector Poisson solve per stage
            w0 = torch.zeros_like(u0)
            rk.op(lgf.OP_CURL, u0, w0)
            w1 = torch.zeros_like(u0)
            return (lambda: rk.step_vorticity(w0, w1, uinf)), [rk], len(xs) * B ** 3, {
                "workload": "one Scheme-A step of the vorticity formulation (Sec. 4.1: curl of the momentum equation, "
                            "velocity by a vector Poisson solve D_supp -> D_xsoln per stage), Re=500 ring, 256^3 box",
                "supp_blocks": int(len(supp)), "xsoln_blocks": int(len(xs)), "points": "D_xsoln points per step",
                "compare": "rk256: the primitive-variable step on the same blocks"}, [t, pv]
        if name == "rk256_refresh":
            return (lambda: rk.refresh(u0, u1)), [rk], len(xs) * B ** 3, {
                "workload": "velocity refresh u = C^T(-L^-1 C u) (vector Poisson D_supp -> D_xsoln), Re=500 ring, "
                            "256^3 bounding box", "supp_blocks": int(len(supp)), "xsoln_blocks": int(len(xs)),
                "qmax_eps_1e-6": rk.qmax(1e-6), "points": "D_xsoln points per refresh"}, [t, pv]
        return (lambda: rk.step(u0, u1, uinf)), [rk], len(xs) * B ** 3, {
            "workload": ("one Scheme-%s IF-HERK step, Re=500 ring (R0 = 50 dx, core 10 dx), 256^3 bounding box, "
                         "D_supp = blocks with |w| > 1e-6 max, D_xsoln = one-block dilation") % "ABC"[scheme],
            "supp_blocks": int(len(supp)), "xsoln_blocks": int(len(xs)), "alpha": dt / (re * dx * dx),
            "points": "D_xsoln points per step"}, [t, pv]
    if name == "vecscal256":
        # vector vs scalar Poisson solve on the 256^3 ring's D_supp -> D_xsoln (the wall-time
        # ratio the paper quotes as ~2.8 for its LGF-FMM; here the three components share
        # every launch of the FFT passes)
        n, R0c, dcells = 256, 50.0, 10.0
        dx = 1.0 / R0c
        axis = inputs.random_axis_tilted(inputs.rng_for(4))
        w = inputs.vortex_ring_edges(n, R0c, dcells, axis) / dx ** 2
        supp = inputs.active_blocks(w, B, 1e-6)
        xs = _dilate(supp)
        t = lgf.Table(lgf.LAPLACE7, max_offset=lgf.required_max_offset(supp, xs, B))
        p1 = lgf.Plan(t, [lgf.Solve(B, 1, supp, xs, dx=dx, scale=-1.0)])
        p3 = lgf.Plan(t, [lgf.Solve(B, 3, supp, xs, dx=dx, scale=-1.0)])
        f3 = torch.from_numpy(inputs.to_blocks(w, B, supp)).cuda()
        f1 = f3[:, :1].contiguous()
        o1 = torch.zeros((len(xs), 1, B, B, B), device="cuda")
        o3 = torch.zeros((len(xs), 3, B, B, B), device="cuda")
        flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")

        def timed_ms(fn, reps=20):
            for _ in range(3):
                fn()
            torch.cuda.synchronize()
            tot = 0.0
            for _ in range(reps):
                flush.fill_(1.0)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                fn()
                b.record()
                torch.cuda.synchronize()
                tot += a.elapsed_time(b)
            return tot / reps
        ms1 = timed_ms(lambda: p1.execute([f1], [o1]))
        ms3 = timed_ms(lambda: p3.execute([f3], [o3]))
        return (lambda: p3.execute([f3], [o3])), [p3], 3 * len(xs) * B ** 3, {
            "workload": "vector (3-component) Poisson solve D_supp -> D_xsoln of the 256^3 Re=500 ring, "
                        "against the scalar solve on the same blocks",
            "supp_blocks": int(len(supp)), "xsoln_blocks": int(len(xs)), "scalar_ms": round(ms1, 4),
            "vector_ms": round(ms3, 4), "vector_to_scalar_ratio": round(ms3 / ms1, 3),
            "points": "3 x D_xsoln points per vector solve"}, [t, p1]
    if name in ("shell256", "shell256_split", "shell256_split_tc"):
        # one scalar Poisson solve D_supp -> D_xsoln of the 256^3 Re = 500 ring shell, by the
        # whole-box FFT convolution or by the block-sparse split solve (FP32 far field on the
        # CUDA cores, or the reduced-precision far field on the tensor cores)
        axis = inputs.random_axis_tilted(inputs.rng_for(4))
        w = inputs.vortex_ring_edges(256, 50.0, 10.0, axis)[0]
        supp = inputs.active_blocks(w, B, 1e-6)
        xs = _dilate(supp)
        method = 0 if name == "shell256" else 1
        K = lgf.required_max_offset(supp, xs, B) if method == 0 else 31
        t = lgf.Table(lgf.LAPLACE7, max_offset=K)
        p = lgf.Plan(t, [lgf.Solve(B, 1, supp, xs, scale=-1.0)], method=method, use_graph=True,
                     far_precision=1 if name.endswith("_tc") else 0)
        f = torch.from_numpy(inputs.to_blocks(w, B, supp)).cuda()
        o = torch.zeros((len(xs), 1, B, B, B), device="cuda")
        return (lambda: p.execute([f], [o])), [p], len(xs) * B ** 3, {
            "workload": "scalar Poisson solve D_supp -> D_xsoln of the 256^3 Re = 500 ring shell (w_x), "
                        + {0: "whole-box FFT convolution", 1: "block-sparse split solve"}[method]
                        + (", far field on the tensor cores (tcgen05, TF32 split)" if name.endswith("_tc") else ""),
            "supp_blocks": int(len(supp)), "xsoln_blocks": int(len(xs)), "points": "D_xsoln points per solve"}, [t]
    if name == "rk_thinring":
        # one Scheme-A IF-HERK step of the delta/R0 = 0.0125 ring (Sec. 6: R0 = 400 cells, core
        # 5 cells, Re = 500, u_inf as for the 256^3 ring), its Poisson solves by the block-sparse
        # split (the box, ~750 cells across, is beyond the whole-box FFT lengths); dt is the 256^3
        # ring's dt Gamma/R0^2 scaled by the cell size and the core radius
        import math
        R0c, dcells = 400.0, 5.0
        dx = 1.0 / R0c
        dt, re = 0.01721 * (50.0 / R0c) * ((dcells / R0c) / 0.2), 500.0
        uinf = (0.0, 0.0, -0.18686)
        supp, w, _ = inputs.thin_ring_vorticity(R0c, dcells, B)
        rk = lgf.RKPlan(B, supp, dx, dt, re, scheme=0, use_graph=True)
        xs = rk.blocks(0)
        pv = lgf.Plan(lgf.Table(lgf.LAPLACE7, max_offset=63), [lgf.Solve(B, 3, supp, xs, dx=dx, scale=-1.0)],
                      method=1)
        a = torch.zeros((len(xs), 3, B, B, B), device="cuda")
        pv.execute([torch.from_numpy(w / dx ** 2).cuda()], [a])
        u0 = torch.zeros_like(a)
        rk.op(lgf.OP_CURL_T, a, u0)
        del a, pv
        # ring speed over 7 steps (outside the timed region) against eq. u_saffman (beta_0 = 0.557966)
        u, v = u0.clone(), torch.zeros_like(u0)
        d0 = rk.diagnostics(u)
        for _ in range(7):
            rk.step(u, v, uinf)
            u, v = v, u
        d1 = rk.diagnostics(u)
        ih = d0["I"] / np.linalg.norm(d0["I"])
        speed = float((d1["X"] - d0["X"]) @ ih / (7 * dt) - np.asarray(uinf) @ ih)
        eps = dcells / R0c
        saffman = (math.log(8 / eps) - 0.557966) / (4 * math.pi)
        u1 = torch.zeros_like(u0)
        del u, v
        return (lambda: rk.step(u0, u1, uinf)), [rk], len(xs) * B ** 3, {
            "workload": "one Scheme-A IF-HERK step of the delta/R0 = 0.0125 ring (R0 = 400 cells, core 5 cells, "
                        "Re = 500), Poisson solves by the block-sparse split solve",
            "supp_blocks": int(len(supp)), "xsoln_blocks": int(len(xs)), "dt": dt, "alpha": dt / (re * dx * dx),
            "ring_speed_vs_saffman": round(speed / saffman - 1, 5), "points": "D_xsoln points per step"}, []
    if name == "thinring_split":
        # the thinnest ring of Sec. 6 (delta / R0 = 0.0125: R0 = 400 cells, core 5 cells), w_x on the
        # blocks above 1e-6 max, targets their one-block dilation: its bounding box (about 750 cells
        # across) is beyond the whole-box embedding's 1024-point FFTs; the split solve runs it
        src_c, vals = inputs.thin_ring_blocks()
        xs = _dilate(src_c)
        t = lgf.Table(lgf.LAPLACE7, max_offset=31)
        p = lgf.Plan(t, [lgf.Solve(B, 1, src_c, xs, scale=-1.0)], method=1, use_graph=True)
        f = torch.from_numpy(vals).cuda()
        o = torch.zeros((len(xs), 1, B, B, B), device="cuda")
        ext = (src_c.max(0) - src_c.min(0) + 1) * B
        return (lambda: p.execute([f], [o])), [p], len(xs) * B ** 3, {
            "workload": "scalar Poisson solve of the delta/R0 = 0.0125 ring (R0 = 400 cells, core 5 cells), "
                        "block-sparse split solve", "supp_blocks": int(len(src_c)), "xsoln_blocks": int(len(xs)),
            "source_extent_cells": [int(e) for e in ext], "points": "D_xsoln points per solve"}, [t]
    if name == "ragged64":
        fs = inputs.ragged_ring_sources(nsolve=64)
        solves, srcs, dsts, pts = [], [], [], 0
        for f in fs:
            sc = inputs.active_blocks(f, B, 1e-14)
            dc = inputs.block_grid(f.shape, B)
            solves.append(lgf.Solve(B, 1, sc, dc, scale=-1.0))
            srcs.append(torch.from_numpy(inputs.to_blocks(f, B, sc)).cuda())
            dsts.append(torch.zeros((len(dc), 1, B, B, B), device="cuda"))
            pts += f.size
        K = max(lgf.required_max_offset(s_.src_blocks, s_.dst_blocks, B) for s_ in solves)
        t = lgf.Table(lgf.LAPLACE7, max_offset=K)
        p = lgf.Plan(t, solves, use_graph=True)
        # the plain form for comparison: one plan per solve, executed one after
        # another on one stream, no graph
        plain = [lgf.Plan(t, [s_]) for s_ in solves]

        def run_plain():
            for pl, a, b in zip(plain, srcs, dsts):
                pl.execute([a], [b])
        plain_ms = _timed_ms(torch, run_plain)
        batched_ms = _timed_ms(torch, lambda: p.execute(srcs, dsts))
        return (lambda: p.execute(srcs, dsts)), [p], pts, {
            "workload": "ragged batch of 64 scalar ring solves, edges 24..192 (log-uniform), one captured graph",
            "points": "sum of e^3 over the batch",
            "plain_ms": round(plain_ms, 4), "batched_ms": round(batched_ms, 4),
            "batched_over_plain": round(plain_ms / batched_ms, 3),
            "plain": "64 single-solve plans executed one after another on one stream, no graph"}, [t]
    raise ValueError(name)


def _timed_ms(torch, fn, reps=20):
    """Mean device time of fn in ms (CUDA events, 256 MiB L2 flush before each rep)."""
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    for _ in range(3):
        fn()
    torch.cuda.synchronize()
    tot = 0.0
    for _ in range(reps):
        flush.fill_(1.0)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        tot += a.elapsed_time(b)
    return tot / reps


def bench_aux(args):
    import torch
    torch.cuda.set_device(0)
    from paper_1601_00035_gb300 import build as libbuild
    libbuild.build()
    from paper_1601_00035_gb300 import lgf
    step, plans, pts, cfg, keep = aux_workload(args.workload, lgf, torch)
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    for _ in range(args.warmup):
        step()
        flush.fill_(1.0)
    torch.cuda.synchronize()
    use_graph = args.workload == "if128"
    graph = None
    if use_graph:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step()
        graph.replay()
        torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    for i in range(args.steps):
        flush.fill_(float(i))
        ev[i][0].record(stream)
        if graph is not None:
            graph.replay()
        else:
            step()
        ev[i][1].record(stream)
    torch.cuda.synchronize()
    ms = [a.elapsed_time(b) for a, b in ev]
    dev_ms = sum(ms)
    # per-kernel shares from a separate profiled pass (not in the timed region)
    for p_ in plans:
        p_.set_profiling(2)
    for _ in range(min(args.steps, 20)):
        step()
    torch.cuda.synchronize()
    kt = {}
    for p_ in plans:
        for k, v in p_.kernel_times().items():
            a = kt.setdefault(k, [0, 0.0])
            a[0] += v[0]
            a[1] += v[1]
        p_.set_profiling(0)
    tot = sum(v[1] for v in kt.values()) or 1.0
    line = {"metric": "Mpoints/s (%s)" % args.workload, "value": round(pts * args.steps / (dev_ms / 1e3) / 1e6, 1),
            "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": round(dev_ms / args.steps, 5), "higher_is_better": True,
            "dtype": "f64" if args.workload.endswith("_f64") else "f32", "data": "synthetic", "config": cfg,
            "kernels": {k: {"launches": v[0], "ms_per_launch": round(v[1] / max(v[0], 1), 5),
                            "share": round(v[1] / tot, 4)} for k, v in kt.items()}}
    print(json.dumps(line))
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--workload", default="ring128",
                    choices=["ring128", "blobs32", "blobs32_f64", "if128", "rk256", "rk256_b", "rk256_c",
                             "rk256_refresh", "vecscal256", "ragged64", "shell256", "shell256_split",
                             "shell256_split_tc", "thinring_split", "rk256_vort", "rk_thinring"],
                    help="ring128 is the headline workload; the others print their own throughput")
    args = ap.parse_args()
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    if args.impl == "reference":
        return bench_reference(args)
    if args.workload != "ring128":
        return bench_aux(args)
    return bench_gpu(args)


if __name__ == "__main__":
    sys.exit(main())
