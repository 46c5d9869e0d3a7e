"""Benchmark of the multiscale debiased Sinkhorn solver on one GB300.

Default line -- the scale workload: 60-D fiber bundles, N = M = 1,000,000
fibers of 20 points per side (20 bundles, features scaled by 1/sqrt(20)),
coarse-to-fine with k-means of 1000 clusters per side, coarse-plan truncation,
eps annealed by q = 0.5 per step (on sigma) down to blur = 2 mm, reach = 20 mm,
FP64 final sums.  One step = one solve of sinkhorn_divergence to its stopping
rule (estimated remaining relative change of S below 1e-6).

`value` is softmin pairs evaluated per second of solve time of the plain
float32 form (CUDA cores; all four symmetric instances, whole solve:
clustering, coarse phase, extrapolation, truncation, fine steps, final sums);
`time_to_solve_ms` its solve time.  The same line carries the tensor-core form
(BF16 hi/lo cross term, FP32 accumulation and log-sum-exp) timed the same way,
and the relative difference of both S from a tightly converged float32 S*.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Other workloads (not the default line; each prints its own JSON line):
    --workload fibers --n N       the same fiber problem at N = M = n
    --workload density            track-density maps (two 64^3 volumes, ~100k voxels, D = 3, grid clusters)
    --workload mlp [--n N]        warm-start network: inference and training throughput
    --workload barycenter         track-density atlas: free-support barycenter of 5 maps
    --workload rates              measured per-clock rates of MUFU ex2 and FP32 FMA (roofline constants)
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

PEAKS_FILE = os.path.join(ROOT, "MEASURED_PEAKS.json")
# Per-SM, per-clock rates on GB300 (sm_103a) used for the ALU bounds: ex2.approx
# 32/clk (the MUFU unit, measured), FP32 128 lanes/clk (f32x2 packing halves
# issue slots, not FP32 work).  A pair of a stable log-sum-exp in the
# dot-product form costs D FMAs, one add (the row's reference), one add
# (accumulate) and one ex2 on the CUDA cores; in the tensor-core forms the
# exponent comes from the tensor core and the CUDA cores keep one ex2 and one
# add per pair.
SFU_EX2_PER_CLK_SM = 32
FP32_LANES_PER_CLK_SM = 128
# tensor flops per pair: D <= 3 float32-accuracy form (K = 32 BF16 slots), the
# 60-D BF16 hi/lo cross term (three K = 64 products), and its float32-accuracy
# form (three pieces per operand, six products)
TC3_TENSOR_FLOP_PER_PAIR = 2 * 32
TC60_TENSOR_FLOP_PER_PAIR = 3 * 2 * 64
FP32_60_TENSOR_FLOP_PER_PAIR = 6 * 2 * 64
# DRAM bytes (ncu dram__bytes_read.sum + dram__bytes_write.sum) per launch of the
# dominant kernel of each workload, from one capture of the current kernel
# (null when the kernel has changed since).
TRAFFIC = {
    "softmin3_tc_kernel": None,
    "softmin_tcc_kernel": None,
}


def peaks():
    return json.load(open(PEAKS_FILE)) if os.path.exists(PEAKS_FILE) else {}


# ------------------------------------------------------------------ inputs --
def fiber_data(n):
    from paper_2107_02010_gb300 import synth

    ctrl = synth.bundle_centrelines()
    x, a, _ = synth.fiber_bundles(n, seed=4, ctrl=ctrl, perturb=3.0)
    y, b, lab = synth.fiber_bundles(n, seed=5, ctrl=ctrl)
    return x, a, y, b


def fiber_params(otgb, n, precision, tol, max_iters):
    # the stopping rule is evaluated every 3 steps (a check costs one FP64 sum
    # and one host read, far below a step of this size)
    return otgb.default_params(blur=2.0, reach=20.0, scaling=0.5, multiscale=1, cluster=1,
                               k_clusters=max(20, n // 1000), kmeans_iters=10, tol=tol, max_iters=max_iters,
                               precision=precision, check_every=3)


def density_data(args):
    from paper_2107_02010_gb300 import synth

    return synth.density_maps(grid=args.grid, n_keep=args.n_keep)


def density_params(args, otgb):
    # the stopping rule is evaluated every 3 steps, as for the fibers (measured at 100k voxels: 91 ms per solve
    # against 101 ms every 10 steps and 108 ms every step; S within 2e-7 of S* either way)
    return otgb.default_params(blur=1.0, reach=10.0, scaling=0.5, multiscale=int(args.multiscale), cluster=0,
                               cell=4.0, tol=args.tol, max_iters=args.max_iters, check_every=3,
                               rows_per_thread=args.rows_per_thread)


# ------------------------------------------------------------------ clocks --
def start_clock_sampler():
    try:
        # the raw samples go to the file named by OTGB_CLOCKS_CSV, if set
        f = open(os.environ.get("OTGB_CLOCKS_CSV") or os.devnull, "a")
        p = subprocess.Popen(
            ["nvidia-smi", "--query-gpu=index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap",
             "--format=csv,noheader,nounits", "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL,
            text=True)
        return p, f
    except Exception:
        return None, None


def stop_clock_sampler(p, f, dev_index=0):
    if p is None:
        return None
    time.sleep(0.3)
    p.terminate()
    try:
        out, _ = p.communicate(timeout=5)
    except Exception:
        p.kill()
        out = ""
    rows = []
    for line in out.splitlines():
        parts = [s.strip() for s in line.split(",")]
        if len(parts) < 9 or parts[0] != str(dev_index):
            continue
        rows.append(parts)
        if f:
            f.write(line + "\n")
    if f:
        f.close()
    if not rows:
        return None
    sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
    mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
    names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
    reasons = sorted({names[k] for r in rows for k in range(4) if r[5 + k].lower() == "active"})
    return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
            "reasons": reasons, "samples": len(rows)}


def flush_l2(buf):
    buf.add_(1.0)  # touches 256 MB (> 129 MB L2)


# ------------------------------------------------------------ CPU baseline --
def oracle_rows_timing(x, y, b, eps, lam, rows, threads=0):
    """Seconds the FP64 oracle takes for the softmin of `rows` rows of x (evenly
    spread) against all columns y (pot = 0), on `threads` threads (0: all)."""
    import oracle

    oracle.build()
    if threads:
        oracle.set_threads(threads)
    pot = np.zeros(y.shape[0])
    idx = np.linspace(0, x.shape[0] - 1, rows).astype(np.int64)
    t0 = time.perf_counter()
    oracle.softmin(x[idx], y, b, pot, eps, lam)
    return time.perf_counter() - t0


def oracle_calibrated(x, y, b, eps, lam, target_s, rows=0, probe=64, threads=0):
    """(rows, seconds): a probe run sets the row count for about target_s."""
    if rows <= 0:
        dt0 = oracle_rows_timing(x, y, b, eps, lam, probe, threads)
        rows = int(min(x.shape[0], max(probe, probe * target_s / max(dt0, 1e-6))))
    return rows, oracle_rows_timing(x, y, b, eps, lam, rows, threads)


def cpu_baseline(x, y, b, eps, lam, label, target_s=10.0, one_core_s=4.0, solve_pairs_dense=None, probe=64):
    """The FP64 oracle's softmin on a bounded sample of the workload, on all the
    host cores and on one core; with solve_pairs_dense (dense pairs of the
    solve: steps x (N^2 + M^2 + 2NM)) the oracle's solve time is extrapolated."""
    import oracle

    oracle.build()
    cores = oracle.threads()
    rows, dt = oracle_calibrated(x, y, b, eps, lam, target_s, probe=probe)
    rate = rows * y.shape[0] / dt
    r1, dt1 = oracle_calibrated(x, y, b, eps, lam, one_core_s, probe=max(4, probe // 8), threads=1)
    oracle.set_threads(cores)
    out = {"value": rate, "unit": "pairs/s", "cores": cores, "kind": "oracle",
           "sample": "FP64 oracle softmin: %d rows x %d columns of the %s (%.1f s on %d threads)" %
                     (rows, y.shape[0], label, dt, cores),
           "one_core": {"value": r1 * y.shape[0] / dt1, "unit": "pairs/s", "cores": 1,
                        "sample": "%d rows x %d columns (%.1f s)" % (r1, y.shape[0], dt1)}}
    if solve_pairs_dense:
        out["extrapolated_solve_s"] = solve_pairs_dense / rate
        out["extrapolated_solve_s_one_core"] = solve_pairs_dense / out["one_core"]["value"]
        out["extrapolation"] = ("extrapolated, not measured: the GPU solve's steps x dense pairs per step "
                                "(N^2 + M^2 + 2NM) / the oracle's pairs/s (the oracle evaluates every pair)")
    return out


# ------------------------------------------------------------------ timing --
def timed_solves(solve, steps, warmup, l2, st):
    """W untimed solves, then K solves each bracketed by CUDA events on the
    launching stream, with a 256 MB write between them (L2 flush)."""
    import torch

    for _ in range(warmup):
        solve()
    torch.cuda.synchronize()
    ms, outs = [], []
    for _ in range(steps):
        flush_l2(l2)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        out = solve()
        e1.record(st)
        e1.synchronize()
        ms.append(e0.elapsed_time(e1))
        outs.append(out)
    torch.cuda.synchronize()
    return ms, outs


def summarize(ms, outs):
    keys = ("prep_ms", "coarse_ms", "fine_ms", "final_ms")
    st = [o["stats"] for o in outs]
    return {
        "time_to_solve_ms": statistics.mean(ms),
        "pairs_per_solve": statistics.mean(s["pairs_evaluated"] for s in st),
        "softmin_ms_per_solve": statistics.mean(s["softmin_ms"] for s in st),
        "iters_per_solve": statistics.mean(s["iters_total"] for s in st),
        "S": outs[-1]["S"],
        "converged": all(o["status"] == 0 for o in outs),
        "phases_ms": {k[:-3]: statistics.mean(s[k] for s in st) for k in keys},
        "kept_fraction": st[-1]["kept_fraction"],
    }


def e2e_solves(solve_host, repeats):
    """End to end through the public API: pinned host inputs copied in, the
    solve, S and the duals f, g read back; wall time per repeat."""
    import torch

    solve_host()  # one untimed pass (same buffers as the timed ones)
    out = []
    for _ in range(repeats):
        torch.cuda.synchronize()
        t1 = time.perf_counter()
        solve_host()
        torch.cuda.synchronize()
        out.append((time.perf_counter() - t1) * 1e3)
    return out


def dist_setup():
    import torch

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    torch.cuda.set_device(local)
    return world, rank, local


def barrier(world):
    import torch

    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()


# ------------------------------------------------------------------ fibers --
def run_fibers(args):
    """60-D fibers, N = M = n: the float32 form (the line's value) and the
    tensor-core form, each W warm-up + K timed solves to the stopping rule."""
    import torch

    world, rank, local = dist_setup()
    from paper_2107_02010_gb300 import otgb, replicas

    n = args.n
    x, a, y, b = fiber_data(n)
    dev = torch.device("cuda", local)
    X, A, Y, B = (torch.from_numpy(v).to(dev) for v in (x, a, y, b))
    ctx = otgb.Context()
    st = torch.cuda.current_stream(dev)
    l2 = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)
    p32 = fiber_params(otgb, n, 0, args.tol, args.max_iters)
    ptc = fiber_params(otgb, n, 1, args.tol, args.max_iters)
    solve32 = lambda: otgb.sinkhorn_divergence(ctx, X, A, Y, B, p32, raise_on_noconv=False)
    solvetc = lambda: otgb.sinkhorn_divergence(ctx, X, A, Y, B, ptc, raise_on_noconv=False)
    D = x.shape[1]
    pk = peaks()
    n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
    clk = pk.get("sm_max_mhz", 2070.0)

    # float32 form: the line's value
    barrier(world)
    sampler, sf = start_clock_sampler()
    l0 = otgb.kernel_launches()
    ms32, outs32 = timed_solves(solve32, args.steps, args.warmup, l2, st)
    launches = otgb.kernel_launches() - l0
    clocks = stop_clock_sampler(sampler, sf, local)
    barrier(world)
    s32 = summarize(ms32, outs32)
    t_total, pairs = replicas.aggregate(sum(ms32) / 1e3, s32["pairs_per_solve"] * args.steps, dev)
    value = pairs / t_total

    # tensor-core form
    tc = None
    if not args.no_tc:
        sampler, sf = start_clock_sampler()
        mstc, outstc = timed_solves(solvetc, args.steps, args.warmup, l2, st)
        clocks_tc = stop_clock_sampler(sampler, sf, local)
        tc = summarize(mstc, outstc)
        tc["clocks"] = clocks_tc
        # the paper's own schedule, q = 0.9 on sigma (Section 2), against the workload's q = 0.5:
        # tensor-core form, one untimed and three timed solves
        pq = fiber_params(otgb, n, 1, args.tol, args.max_iters)
        pq.scaling = 0.9
        msq, outsq = timed_solves(lambda: otgb.sinkhorn_divergence(ctx, X, A, Y, B, pq, raise_on_noconv=False),
                                  3, 1, l2, st)
        tc["q_0.9"] = summarize(msq, outsq)

    # S* of the stopping-rule check: one tightly converged float32 solve (untimed)
    # (at least 60 steps at blur, past the point where the float32 iteration stops contracting)
    pref = fiber_params(otgb, n, 0, 1e-9, 20000)
    pref.min_iters = 60
    ref = otgb.sinkhorn_divergence(ctx, X, A, Y, B, pref, raise_on_noconv=False)
    S_star = ref["S"]

    # end to end through the public API from pinned host buffers
    hx, ha, hy, hb = (torch.from_numpy(v).pin_memory() for v in (x, a, y, b))

    def solve_host():
        Xd, Ad, Yd, Bd = (h.to(dev, non_blocking=True) for h in (hx, ha, hy, hb))
        o = otgb.sinkhorn_divergence(ctx, Xd, Ad, Yd, Bd, p32, raise_on_noconv=False)
        o["f"].cpu(), o["g"].cpu()
        return o

    e2e_ms = e2e_solves(solve_host, max(1, min(args.steps, args.e2e_steps)))
    e2e_val = s32["pairs_per_solve"] / (statistics.mean(e2e_ms) / 1e3) * max(world, 1)
    h2d = sum(v.nbytes for v in (x, a, y, b))
    d2h = 4 * (x.shape[0] + y.shape[0])

    # roofline of the dominant kernel (softmin_tcc_kernel, three BF16 pieces per operand: float32 accuracy)
    peak = min(pk.get("bf16_tflops", 1910.7) * 1e12 / FP32_60_TENSOR_FLOP_PER_PAIR, SFU_EX2_PER_CLK_SM * n_sm * clk * 1e6)
    achieved = s32["pairs_per_solve"] / (s32["softmin_ms_per_solve"] / 1e3)
    line = {
        "metric": "softmin pairs/s", "value": value, "unit": "pairs/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": s32["time_to_solve_ms"], "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "60-D fiber bundles (20 points x 3-D, scaled 1/sqrt(20)), 20 bundles, N=M=%d, "
                               "k-means %d clusters per side, coarse-plan truncation, blur 2 mm, reach 20 mm, "
                               "q 0.5, FP64 final sums, stop at est. rel. change of S < %g" %
                               (n, max(20, n // 1000), args.tol),
                   "N": n, "M": n, "D": D,
                   "l2": "inputs larger than L2 (240 MB per side); 256 MB buffer written between timed steps",
                   "parallelism": "replicas" if world > 1 else "1 GPU"},
        "time_to_solve_ms": s32["time_to_solve_ms"],
        "S": s32["S"], "S_star": S_star, "rel_err_S": abs(s32["S"] - S_star) / abs(S_star),
        "S_star_from": "float32 solve to est. rel. change < 1e-9, at least 60 steps at blur (%d steps)" %
                       ref["stats"]["iters_total"],
        "converged": s32["converged"], "iters_per_solve": s32["iters_per_solve"],
        "pairs_per_solve": s32["pairs_per_solve"], "kept_fraction": s32["kept_fraction"],
        "softmin_ms_per_solve": s32["softmin_ms_per_solve"], "phases_ms": s32["phases_ms"],
        "roofline": {"bound": "tensor", "kernel": "softmin_tcc_kernel (three-piece BF16 operands, float32 accuracy)",
                     "achieved": achieved / 1e9, "peak": peak / 1e9, "unit": "Gpairs/s", "frac": achieved / peak,
                     "traffic": TRAFFIC["softmin_tcc_kernel"],
                     "peak_basis": "bf16 burst of measured / %d flop per pair; MUFU ex2 (32/clk) is not binding" %
                                   FP32_60_TENSOR_FLOP_PER_PAIR},
        "e2e": {"value": e2e_val, "unit": "pairs/s", "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                "repeats": len(e2e_ms), "ms_per_step": statistics.mean(e2e_ms)},
        "gpu_launches": int(launches), "clocks": clocks,
    }
    if tc is not None:
        peak_tc = min(pk.get("bf16_tflops", 1910.7) * 1e12 / TC60_TENSOR_FLOP_PER_PAIR,
                      SFU_EX2_PER_CLK_SM * n_sm * clk * 1e6)
        ach_tc = tc["pairs_per_solve"] / (tc["softmin_ms_per_solve"] / 1e3)
        tc["q_0.9"]["rel_err_S"] = abs(tc["q_0.9"]["S"] - S_star) / abs(S_star)
        tc.update({"dtype": "bf16 hi/lo cross term (three products), f32 accumulate, f32 log-sum-exp",
                   "rel_err_S": abs(tc["S"] - S_star) / abs(S_star),
                   "speedup_vs_fp32": s32["time_to_solve_ms"] / tc["time_to_solve_ms"],
                   "value": tc["pairs_per_solve"] / (tc["time_to_solve_ms"] / 1e3),
                   "roofline": {"bound": "tensor", "kernel": "softmin_tcc_kernel (cluster-tiled tcgen05 form)",
                                "achieved": ach_tc / 1e9, "peak": peak_tc / 1e9, "unit": "Gpairs/s",
                                "frac": ach_tc / peak_tc,
                                "peak_basis": "bf16 burst of measured / %d flop per pair" %
                                              TC60_TENSOR_FLOP_PER_PAIR}})
        line["tensor_core_form"] = tc
    if not args.no_cpu_baseline and world <= 1:
        dense = (2.0 * n * n + 2.0 * n * n) * s32["iters_per_solve"]
        line["cpu_baseline"] = cpu_baseline(x, y, b, 4.0, 1.0 / 1.01, "60-D fiber workload", target_s=10.0,
                                            one_core_s=4.0, solve_pairs_dense=dense, probe=16)
    if rank == 0:
        print(json.dumps(line))
    ctx.close()
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


# ----------------------------------------------------------------- density --
def run_density(args):
    """Track-density maps (D = 3, grid clusters): one solve per step."""
    import torch

    world, rank, local = dist_setup()
    from paper_2107_02010_gb300 import otgb, replicas

    x, a, y, b = density_data(args)
    dev = torch.device("cuda", local)
    X, A, Y, B = (torch.from_numpy(v).to(dev) for v in (x, a, y, b))
    ctx = otgb.Context()
    p = density_params(args, otgb)
    st = torch.cuda.current_stream(dev)
    l2 = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)
    solve = lambda: otgb.sinkhorn_divergence(ctx, X, A, Y, B, p, raise_on_noconv=False)
    barrier(world)
    sampler, sf = start_clock_sampler()
    l0 = otgb.kernel_launches()
    ms, outs = timed_solves(solve, args.steps, args.warmup, l2, st)
    launches = otgb.kernel_launches() - l0
    clocks = stop_clock_sampler(sampler, sf, local)
    barrier(world)
    s = summarize(ms, outs)
    t_total, pairs = replicas.aggregate(sum(ms) / 1e3, s["pairs_per_solve"] * args.steps, dev)
    hx, ha, hy, hb = (torch.from_numpy(v).pin_memory() for v in (x, a, y, b))

    def solve_host():
        Xd, Ad, Yd, Bd = (h.to(dev, non_blocking=True) for h in (hx, ha, hy, hb))
        o = otgb.sinkhorn_divergence(ctx, Xd, Ad, Yd, Bd, p, raise_on_noconv=False)
        o["f"].cpu(), o["g"].cpu()

    e2e_ms = e2e_solves(solve_host, args.steps)
    # S* for the accuracy of the timed solves: the same problem to est. rel. change < 1e-9
    pstar = density_params(args, otgb)
    pstar.tol = 1e-9
    pstar.max_iters = max(args.max_iters, 20000)
    S_star = otgb.sinkhorn_divergence(ctx, X, A, Y, B, pstar, raise_on_noconv=False)["S"]
    pk = peaks()
    n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
    clk = pk.get("sm_max_mhz", 2070.0)
    # the default D <= 3 kernel (softmin3_tc_kernel): min(MUFU ex2, tensor pipe)
    peak_mufu = SFU_EX2_PER_CLK_SM * n_sm * clk * 1e6
    peak_tensor = pk.get("bf16_tflops", 1910.7) * 1e12 / TC3_TENSOR_FLOP_PER_PAIR
    peak = min(peak_mufu, peak_tensor)
    achieved = s["pairs_per_solve"] / (s["softmin_ms_per_solve"] / 1e3)
    line = {
        "metric": "softmin pairs/s", "workload": "density", "value": pairs / t_total, "unit": "pairs/s",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": s["time_to_solve_ms"],
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "bf16x3 three-piece exponent on the tensor cores (float32 accuracy), f32 sums",
        "data": "synthetic",
        "config": {"workload": "track-density maps: two 64^3 volumes of 30 Gaussian tubes, %d voxels per side, "
                               "masses 1.0/1.2, p=2, blur=1, reach=10, q=0.5, multiscale grid cells of 4 voxels, "
                               "stop at est. rel. change of S < %g" % (x.shape[0], args.tol),
                   "N": int(x.shape[0]), "M": int(y.shape[0]), "D": 3,
                   "l2": "256 MB buffer written between timed steps (inputs are smaller than L2)",
                   "parallelism": "replicas" if world > 1 else "1 GPU"},
        **s,
        "S_star": S_star, "rel_err_S": abs(s["S"] - S_star) / abs(S_star),
        "S_star_from": "the same solve to est. rel. change < 1e-9",
        "roofline": {"bound": "alu", "kernel": "softmin3_tc_kernel (+ fallback)", "achieved": achieved / 1e9,
                     "peak": peak / 1e9, "unit": "Gpairs/s", "frac": achieved / peak,
                     "traffic": TRAFFIC["softmin3_tc_kernel"],
                     "peak_basis": "MUFU ex2: %d SMs x 32 ex2/clk x %.0f MHz, below the tensor bound %.3g pairs/s "
                                   "(bf16 of measured, %d flop per pair)" % (n_sm, clk, peak_tensor,
                                                                            TC3_TENSOR_FLOP_PER_PAIR)},
        "e2e": {"value": s["pairs_per_solve"] / (statistics.mean(e2e_ms) / 1e3) * max(world, 1), "unit": "pairs/s",
                "h2d_bytes_per_step": sum(v.nbytes for v in (x, a, y, b)),
                "d2h_bytes_per_step": 4 * (x.shape[0] + y.shape[0])},
        "gpu_launches": int(launches), "clocks": clocks,
    }
    if not args.no_cpu_baseline and world <= 1:
        line["cpu_baseline"] = cpu_baseline(x, y, b, 1.0, 1.0 / 1.01, "track-density workload", target_s=10.0,
                                            one_core_s=4.0, probe=2048)
    if rank == 0:
        print(json.dumps(line))
    ctx.close()
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


# ------------------------------------------------------------------- rates --
def run_rates(args):
    """Measured per-SM, per-clock unit rates (otgb_unit_rates): MUFU ex2,
    scalar FP32 FMA, packed FP32x2 FMA -- the constants of the ALU rooflines."""
    import torch
    from paper_2107_02010_gb300 import otgb

    ctx = otgb.Context()
    vals = [otgb.unit_rates(ctx) for _ in range(max(1, args.steps))]
    med = {k: statistics.median(v[k] for v in vals) for k in vals[0]}
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    print(json.dumps({"metric": "unit rates", "workload": "rates", "unit": "lane operations per clock per SM",
                      "ex2": med["ex2"], "fma": med["fma"], "fma2": med["fma2"], "repeats": len(vals),
                      "n_sm": n_sm, "used_by_roofline": {"ex2": SFU_EX2_PER_CLK_SM, "fma": FP32_LANES_PER_CLK_SM}}))
    return 0


# -------------------------------------------------------------- barycenter --
def run_barycenter(args):
    """Track-density atlas: the free-support barycenter of K = 5 unit-mass
    density maps of 20,000 voxels (64^3 volumes), initialised with their
    average density up-sampled 6 times; blur 1 voxel, reach = inf, p = 2,
    multiscale grid cells of 4 voxels.  One step = one barycenter of `--iters`
    gradient steps (lr = 1), each from K solves and K gradients.  The solves stop
    at tol = 1e-4 (checked every 3 steps): the objective after each gradient
    step then matches that of tol = 1e-6 solves to about 5e-6 relative, in
    half the time."""
    import torch
    from paper_2107_02010_gb300 import otgb, synth

    x0, a0, ys, bs = synth.barycenter_maps()
    ctx = otgb.Context()
    A0, X0 = torch.from_numpy(a0).cuda(), torch.from_numpy(x0).cuda()
    Ys = [torch.from_numpy(y).cuda() for y in ys]
    Bs = [torch.from_numpy(b).cuda() for b in bs]
    p = otgb.default_params(blur=1.0, reach=0.0, scaling=0.5, multiscale=1, cluster=0, cell=4.0, tol=1e-4,
                            max_iters=5000, check_every=3)
    st = torch.cuda.current_stream()
    l2 = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")

    def solve():
        X = X0.clone()
        return otgb.sinkhorn_barycenter(ctx, X, A0, Ys, Bs, p, iters=args.iters, lr=1.0), X

    l0 = otgb.kernel_launches()
    ms, outs = [], []
    for k in range(args.warmup + args.steps):
        flush_l2(l2)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        hist, X = solve()
        e1.record(st)
        e1.synchronize()
        if k >= args.warmup:
            ms.append(e0.elapsed_time(e1))
    line = {"metric": "barycenter time", "workload": "barycenter", "value": statistics.mean(ms) / 1e3, "unit": "s",
            "steps": args.steps, "warmup": args.warmup, "higher_is_better": False, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": "free-support Sinkhorn barycenter of 5 track-density maps (64^3, 20,000 voxels, "
                                   "unit mass), %d support points (average density up-sampled x6), blur 1 voxel, "
                                   "reach inf, grid cells of 4 voxels, %d gradient steps, solves to tol 1e-4" % (
                                       x0.shape[0], args.iters)},
            "objective": hist, "gpu_launches": int(otgb.kernel_launches() - l0),
            "paper_context": "about 9 s on a GTX 1080 for ~400,000 support points and 5 maps of ~20,000 voxels "
                             "(Section 3, track density atlas); other hardware, context only"}
    print(json.dumps(line))
    return 0


# -------------------------------------------------------------------- warm --
def run_warm(args):
    """Learned warm start against a fixed atlas, time-to-solve: a 300k-fiber
    atlas; `--warm-train` training subjects and `--warm-test` test subjects of
    uneven sizes (uniform in [100k, 400k] fibers, each subject's bundles
    displaced by its own perturbation); the network (60 -> 256 -> 256 -> 256 ->
    1) trained on the f potentials of plain solves of the training subjects.
    One step = every test subject solved by the plain multiscale FP32 form and
    by the warm-started form, both with the stopping rule tol = 1e-4 checked
    every 3 steps (the S they return is checked against a tight reference
    solve, tol 1e-9, at 1e-5 relative).  Times are device times of the solves (the warm one including
    the network's inference)."""
    import torch
    from paper_2107_02010_gb300 import otgb, synth

    BLUR, REACH = 2.0, 20.0

    def P(n, **kw):
        base = dict(blur=BLUR, reach=REACH, scaling=0.5, multiscale=1, cluster=1, k_clusters=1000,
                    kmeans_iters=10, tol=1e-4, max_iters=3000, check_every=3)
        base.update(kw)
        return otgb.default_params(**base)

    t_start = time.time()
    ctx = otgb.Context()
    ctrl = synth.bundle_centrelines()
    y, b, _ = synth.fiber_bundles(300000, seed=10, ctrl=ctrl)
    yt, bt = torch.from_numpy(y).cuda(), torch.from_numpy(b).cuda()
    rng = np.random.default_rng(0)
    X, F = [], []
    b_atlas = None
    for s in range(args.warm_train):
        n = int(rng.integers(100000, 400001))
        x, a, _ = synth.fiber_bundles(n, seed=100 + s, ctrl=ctrl, perturb=3.0)
        xt, at = torch.from_numpy(x).cuda(), torch.from_numpy(a).cuda()
        r = otgb.sinkhorn_divergence(ctx, xt, at, yt, bt, P(n, tol=1e-8), want_self=True)
        X.append(xt)
        F.append(r["f"])
        if b_atlas is None:
            b_atlas = r["b_self"].clone()
    Xc, Fc = torch.cat(X), torch.cat(F)
    t_targets = time.time() - t_start
    net = otgb.Mlp(ctx, 60, 256, seed=7)
    net.fit_normalization(Xc, Fc)
    losses = []
    torch.cuda.synchronize()
    t0 = time.time()
    for e in range(args.warm_epochs):
        lr = 1e-5 + 0.5 * (1e-3 - 1e-5) * (1 + np.cos(np.pi * e / args.warm_epochs))
        losses.append(net.train_epoch(Xc, Fc, 16384, lr, seed=e))
    torch.cuda.synchronize()
    t_train = time.time() - t0
    tests = []
    f0_err = []
    for s in range(args.warm_test):
        n = int(rng.integers(100000, 400001))
        x, a, _ = synth.fiber_bundles(n, seed=300 + s, ctrl=ctrl, perturb=3.0)
        xt, at = torch.from_numpy(x).cuda(), torch.from_numpy(a).cuda()
        ref = otgb.sinkhorn_divergence(ctx, xt, at, yt, bt, P(n, tol=1e-9, max_iters=6000))
        f0_err.append(float((net.infer(xt) - ref["f"]).abs().median()) / (BLUR ** 2))
        tests.append((n, xt, at, ref))
    l0 = otgb.kernel_launches()
    acc = {"plain": [0, 0.0, 0.0], "warm": [0, 0.0, 0.0]}
    fell_back = 0
    for k in range(args.warmup + args.steps):
        for n, xt, at, ref in tests:
            rp = otgb.sinkhorn_divergence(ctx, xt, at, yt, bt, P(n))
            rw = otgb.sinkhorn_divergence_warm(ctx, net, xt, at, yt, bt, P(n), b_atlas=b_atlas)
            if k < args.warmup:
                continue
            fell_back += int(rw["stats"]["warm_start"] == 2)
            for key, r, ms in (("plain", rp, rp["stats"]["total_ms"]), ("warm", rw, rw["stats"]["warm_ms"])):
                acc[key][0] += r["stats"]["iters_total"]
                acc[key][1] += ms
                acc[key][2] = max(acc[key][2], abs(r["S"] - ref["S"]) / abs(ref["S"]))
    ns = args.steps * len(tests)
    warm_s = acc["warm"][1] / ns / 1e3
    plain_s = acc["plain"][1] / ns / 1e3
    line = {"metric": "time-to-solve, learned warm start", "workload": "warm", "value": warm_s, "unit": "s",
            "steps": args.steps, "warmup": args.warmup, "higher_is_better": False, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": "learned warm start against a fixed 300k-fiber atlas (60-D fibers, blur 2, reach 20, "
                                   "k-means 1000 clusters); %d training and %d test subjects of 100k-400k fibers; "
                                   "network 60-256-256-256-1 trained %d epochs" % (
                                       args.warm_train, args.warm_test, args.warm_epochs)},
            "per_subject": {"plain_s": plain_s, "warm_s": warm_s, "plain_steps": acc["plain"][0] / ns,
                            "warm_steps": acc["warm"][0] / ns, "plain_max_rel_S_err": acc["plain"][2],
                            "warm_max_rel_S_err": acc["warm"][2], "warm_fell_back": fell_back},
            "plain_over_warm": plain_s / warm_s,
            "f0_median_abs_err_in_eps": f0_err, "train_loss_first_last": [losses[0], losses[-1]],
            "targets_s": t_targets, "training_s": t_train,
            "gpu_launches": int(otgb.kernel_launches() - l0)}
    print(json.dumps(line))
    return 0


# --------------------------------------------------------------------- mlp --
def run_mlp(args):
    """Warm-start network throughput: inference over n rows and one training
    epoch over n rows (batches of `--train-batch`, default 16384), FLOPs
    counted as 2 per multiply-add of the four layers (input padded to 64);
    training = 3 x forward."""
    import torch
    from paper_2107_02010_gb300 import otgb

    ctx = otgb.Context()
    D, H = 60, 256
    net = otgb.Mlp(ctx, D, H, seed=1)
    r = np.random.default_rng(0)
    n = args.n
    x = torch.from_numpy(r.normal(0, 1, (n, D)).astype(np.float32)).cuda()
    f = torch.from_numpy(r.normal(0, 1, n).astype(np.float32)).cuda()
    fwd = 2.0 * n * (64 * H + 2 * H * H + H)
    tb = args.train_batch
    for _ in range(args.warmup):
        net.infer(x)
        net.train_epoch(x, f, tb, 1e-4, seed=0)
    torch.cuda.synchronize()
    st = torch.cuda.current_stream()
    l0 = otgb.kernel_launches()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
    ev[0].record(st)
    for _ in range(args.steps):
        net.infer(x)
    ev[1].record(st)
    ev[2].record(st)
    for k in range(args.steps):
        net.train_epoch(x, f, tb, 1e-4, seed=k + 1)
    ev[3].record(st)
    torch.cuda.synchronize()
    inf_ms = ev[0].elapsed_time(ev[1]) / args.steps
    tr_ms = ev[2].elapsed_time(ev[3]) / args.steps
    peak = peaks().get("bf16_tflops", 1910.7)
    line = {"metric": "warm-start network TFLOP/s", "workload": "mlp", "unit": "TFLOP/s",
            "value": fwd / inf_ms / 1e9, "steps": args.steps, "warmup": args.warmup, "dtype": "bf16",
            "data": "synthetic", "higher_is_better": True,
            "config": {"workload": "MLP %d->%d->%d->%d->1 SiLU, %d rows" % (D, H, H, H, n), "train_batch": tb},
            "inference_ms": inf_ms, "inference_tflops": fwd / inf_ms / 1e9,
            "train_epoch_ms": tr_ms, "train_tflops": 3 * fwd / tr_ms / 1e9,
            "roofline": {"bound": "tensor", "peak": peak, "unit": "TFLOP/s",
                         "frac_inference": fwd / inf_ms / 1e9 / peak, "frac_train": 3 * fwd / tr_ms / 1e9 / peak,
                         "peak_basis": "bf16 burst, of measured"},
            "gpu_launches": int(otgb.kernel_launches() - l0)}
    print(json.dumps(line))
    return 0


# --------------------------------------------------------------- reference --
def run_reference(args):
    """The reference arm: the FP64 oracle timed on the host cores, each step a
    bounded sample of the same workload (rows of the beta -> alpha softmin
    against all columns), calibrated once to about 5 s of host work."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    if args.workload == "density":
        x, a, y, b = density_data(args)
        eps, label, probe = 1.0, "track-density maps 64^3, ~%d voxels per side" % x.shape[0], 2048
    else:
        x, a, y, b = fiber_data(args.n)
        eps, label, probe = 4.0, "60-D fiber bundles, N=M=%d" % args.n, 16
    lam = 1.0 / 1.01
    rows = args.ref_rows
    vals, last = [], None
    for k in range(args.warmup + args.steps):
        rows, dt = oracle_calibrated(x, y, b, eps, lam, 5.0, rows=rows, probe=probe)
        if k >= args.warmup:
            vals.append(rows * y.shape[0] / dt)
            last = (rows, dt)
    import oracle

    v = statistics.mean(vals)
    line = {"impl": "reference", "metric": "softmin pairs/s", "value": v, "unit": "pairs/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": label + ", FP64 oracle softmin sample"},
            "cpu_baseline": {"value": v, "unit": "pairs/s", "cores": oracle.threads(), "kind": "oracle",
                             "sample": "FP64 oracle softmin: %d rows x %d columns per step (%.1f s)" %
                                       (last[0], y.shape[0], last[1])},
            "e2e": {"value": v, "unit": "pairs/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="fibers",
                    choices=["fibers", "density", "mlp", "barycenter", "rates", "warm"])
    ap.add_argument("--warm-train", type=int, default=8)
    ap.add_argument("--warm-test", type=int, default=3)
    ap.add_argument("--warm-epochs", type=int, default=30)
    ap.add_argument("--train-batch", type=int, default=16384)
    ap.add_argument("--iters", type=int, default=5, help="barycenter: gradient steps")
    ap.add_argument("--n", type=int, default=0, help="fibers: points per side (1,000,000); mlp: rows (1,048,576)")
    ap.add_argument("--grid", type=int, default=64)
    ap.add_argument("--n-keep", type=int, default=100_000)
    ap.add_argument("--multiscale", type=int, default=1)
    # the stopping rule: estimated relative change of S below tol (1e-5, the accuracy the time-to-solve is quoted
    # at; the S it returns is within about 1e-7 of the converged S* on the fiber workload)
    ap.add_argument("--tol", type=float, default=1e-5)
    ap.add_argument("--max-iters", type=int, default=5000)
    ap.add_argument("--ref-rows", type=int, default=0, help="oracle sample rows (0: calibrated to about 5 s)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-tc", action="store_true", help="fibers: skip the tensor-core form")
    ap.add_argument("--e2e-steps", type=int, default=3, help="fibers: end-to-end repeats")
    ap.add_argument("--rows-per-thread", type=int, default=0)
    args = ap.parse_args()
    if args.workload == "fibers":
        args.n = args.n or 1_000_000
    elif args.workload == "mlp":
        args.n = args.n or (1 << 20)
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "density":
        return run_density(args)
    if args.workload == "mlp":
        return run_mlp(args)
    if args.workload == "barycenter":
        return run_barycenter(args)
    if args.workload == "rates":
        return run_rates(args)
    if args.workload == "warm":
        return run_warm(args)
    return run_fibers(args)


if __name__ == "__main__":
    sys.exit(main())
