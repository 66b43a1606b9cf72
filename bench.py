"""Benchmark: HOTRG coarse-graining steps/s on one GB300 (per rank).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--precision bf16x6|bf16x3|tf32x3|tf32|fp64]
                    [--workload ising3d_chi16|ising3d_chi20|ising4d_chi6|ising4d_chi13|ising4d_chi14|
                                batch3d_mixed|energy3d_chi12|energy3d_chi12_scan]
                    [--z2 on|off] [--shard] [--impl ours|reference]

Default workload: 3D Ising, d = 3, chi = 16, beta = 0.2216544, h = 0, axes cycling
z, x, y.  The first steps grow the bonds (2 -> 4 -> 16 for the default) and are not
timed; then W steady-state warm-up steps and K timed steps, each one full
coarse-graining (permutation, FP64 environments, eigen-solver, choice/truncation, prime
chain, bottleneck, non-prime chain, trace/normalisation).  The local tensor (134 MB
FP64 for the default) and the per-slice operands (GBs) exceed the 129 MB L2.
Per-step ln Z/V is compared with the FP64 oracle's reference values in
tests/golden/<workload>.jsonl where those exist.

Other workloads: the paper-shape 4D steps (ising4d_chi13/14), the batching form
(batch3d_mixed: 64 independent instances stepped together) and the differentiation form
(energy3d_chi12: steps carrying d/d beta, the internal energy checked against central
differences of FP64 runs; energy3d_chi12_scan: 32 beta in [0.21, 0.23] with energy and
specific heat).

Multi-GPU: independent replicas (one run per rank), weak scaling, no
collective on the data path; rank 0 prints one JSON line.  With --shard every
rank takes part in ONE run instead: each step is split by c'-slices over the
ranks (paper_2110_03607_gb300/shard.py: this rank's part of the environment
Grams, an NCCL all_reduce, the isometries, this rank's c'-slices of the new
tensor, an NCCL all_gather), strong scaling; at N = 1 it runs over a
one-rank NCCL group.
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

METRIC = "3D-Ising chi=16 HOTRG steps/s, split-BF16 vs FP64, rel err in f<=1e-7; TFLOP/s"

# workload -> lattice dimension, bond dimension, coupling, field, first axis, the number of
# bond-growth steps before every bond reaches chi (not timed), and a description
WORKLOADS = {
    "ising3d_chi16": dict(d=3, chi=16, beta=0.2216544, h=0.0, first=2, growth=3,
                          text="3D Ising HOTRG d=3 chi=16 beta=0.2216544 h=0, axes z,x,y"),
    "ising3d_chi20": dict(d=3, chi=20, beta=0.2216544, h=0.0, first=2, growth=5,
                          text="3D Ising HOTRG d=3 chi=20 beta=0.2216544 h=0, axes z,x,y"),
    "ising4d_chi6": dict(d=4, chi=6, beta=0.15, h=0.0, first=0, growth=3,
                         text="4D Ising HOTRG d=4 chi=6 beta=0.15 h=0, axes x,y,z,w"),
    # the shape of the paper's own timing runs (Sec. 5: 4D Ising, chi = 13 and 14)
    "ising4d_chi13": dict(d=4, chi=13, beta=0.15, h=0.0, first=0, growth=4,
                          text="4D Ising HOTRG d=4 chi=13 beta=0.15 h=0, axes x,y,z,w"),
    "ising4d_chi14": dict(d=4, chi=14, beta=0.15, h=0.0, first=0, growth=4,
                          text="4D Ising HOTRG d=4 chi=14 beta=0.15 h=0, axes x,y,z,w"),
    # batching form: independent 3D instances, 16 per chi in {6, 8, 10, 12}, beta uniform
    # in [0.20, 0.24], h alternating 0 / 0.01, stepped together
    "batch3d_mixed": dict(d=3, chi=12, beta=0.22, h=0.0, first=2, growth=3,
                          text="batching form: 64 independent 3D Ising HOTRG instances, chi in "
                               "{6,8,10,12} x 16, beta uniform in [0.20,0.24], h in {0,0.01}, axes z,x,y"),
    # differentiation form: d/d beta carried through every step (FP64 dense form), the
    # internal energy per site; checked against central differences of FP64 runs
    "energy3d_chi12": dict(d=3, chi=12, beta=0.22, h=0.0, first=2, growth=3,
                           text="differentiation form: 3D Ising HOTRG d=3 chi=12 beta=0.22 h=0 with "
                                "d/d beta in forward mode (internal energy), axes z,x,y"),
    # the same over a scan of 32 beta in [0.21, 0.23], stepped together (batching form):
    # energy and specific heat per site as functions of beta
    "energy3d_chi12_scan": dict(d=3, chi=12, beta=0.22, h=0.0, first=2, growth=3,
                                text="differentiation form, beta scan: 32 3D Ising HOTRG instances d=3 "
                                     "chi=12 h=0, beta uniform in [0.21,0.23], d/d beta in forward mode, "
                                     "axes z,x,y"),
}


def batch_instances():
    """(beta, h, chi) of the 64 instances of the batching form."""
    out = []
    for chi in (6, 8, 10, 12):
        for i in range(16):
            out.append((0.20 + 0.04 * i / 15.0, 0.0 if i % 2 == 0 else 0.01, chi))
    return out
W = dict(WORKLOADS["ising3d_chi16"])
WORKLOAD = "ising3d_chi16"
D, CHI, BETA, H = W["d"], W["chi"], W["beta"], W["h"]
FIRST_AXIS, GROWTH_STEPS = W["first"], W["growth"]


def max_over_ranks(ms, dist=None, device="cpu"):
    """The slowest rank's time (a plain float without a process group)."""
    if dist is None:
        return float(ms)
    import torch
    t = torch.tensor([float(ms)], device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(steps_per_rank, world, elapsed_ms):
    """Replicas: every rank runs its own steps; whole-job steps/s over the slowest rank."""
    return world * steps_per_rank / (elapsed_ms / 1000.0)


def select_workload(name):
    global W, WORKLOAD, D, CHI, BETA, H, FIRST_AXIS, GROWTH_STEPS
    W = dict(WORKLOADS[name])
    WORKLOAD = name
    D, CHI, BETA, H = W["d"], W["chi"], W["beta"], W["h"]
    FIRST_AXIS, GROWTH_STEPS = W["first"], W["growth"]


def axes_for(n):
    return [(FIRST_AXIS + s) % D for s in range(n)]


# --precision: binding constant, piece products (terms) per algorithmic product, the
# tensor-core rate of the piece type relative to BF16 (TF32 at the recipe's nominal
# 1.1 / 2.25 PFLOP/s dense), and the JSON dtype
PRECISIONS = {
    "bf16x6": ("PREC_BF16X6", 6, 1.0, "bf16x6-split/fp32-acc; f64 env, eig, lnZ"),
    "bf16x3": ("PREC_BF16X3", 3, 1.0, "bf16x3-split/fp32-acc; f64 env, eig, lnZ"),
    "tf32x3": ("PREC_TF32X3", 3, 1.1 / 2.25, "tf32x3-split/fp32-acc; f64 env, eig, lnZ"),
    "tf32": ("PREC_TF32", 1, 1.1 / 2.25, "tf32/fp32-acc; f64 env, eig, lnZ"),
    "fp64": ("PREC_FP64", 1, None, "f64"),
}


def prec_const(pkg, name):
    return getattr(pkg, PRECISIONS[name][0])


FP64_DIGIT_PRODUCTS = 44   # BF16 products in one FP64 product on the tensor cores: 43 of digits, one for its guard


def fp64_peak(pkg):
    """(TFLOP/s, its source): large FP64 products run as digit products on the tensor cores, the small
    ones on the FP64 pipe; the higher of the two rates bounds both."""
    pipe = pkg.hotrg_fp64_rate()
    peaks, src = load_peaks()
    digits = float(peaks.get("bf16_tflops_sustained", 1700.0)) / FP64_DIGIT_PRODUCTS
    if digits > pipe:
        return digits, f"bf16_tflops_sustained of {src} / {FP64_DIGIT_PRODUCTS} digit products"
    return pipe, "FP64 FMA rate measured in this run (hotrg_fp64_rate)"


def load_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}, "fallback"


def load_golden():
    path = os.path.join(ROOT, "tests", "golden", WORKLOAD + ".jsonl")
    out = {}
    try:
        with open(path) as f:
            for line in f:
                r = json.loads(line)
                if r.get("kind") == "step":
                    out[r["step"]] = r["ln_z_per_site"]
    except OSError:
        pass
    return out


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms."""

    def __init__(self, index: int):
        self.index = index
        self.rows = []
        self.proc = None

    def start(self):
        cmd = ["nvidia-smi", f"--id={self.index}",
               "--query-gpu=clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
               "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
               "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap",
               "--format=csv,noheader,nounits", "-lms", "200"]
        try:
            self.proc = subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        threading.Thread(target=self._read, daemon=True).start()

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 8:
                self.rows.append(parts)

    def stop(self):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        if not self.rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        sm = [float(r[0]) for r in self.rows if r[0].replace(".", "").isdigit()]
        smax = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = set()
        for r in self.rows:
            for k, nm in enumerate(names):
                if r[4 + k].lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(self.rows)}


# ---------------------------------------------------------------------------
# the oracle legs (CPU): bounded samples of one steady-state step
# ---------------------------------------------------------------------------

def oracle_steady_tensor():
    from oracle import hotrg_oracle as o
    run = o.HotrgRun(D, BETA, H)
    for a in axes_for(GROWTH_STEPS):
        run.step(a, CHI)
    return run


def oracle_step_sample(run, axis, sample_iters):
    """Time one oracle step on a sample: environments + eigen-solver in full,
    `sample_iters` of the (c'_0, n') contraction iterations; return the
    extrapolated seconds of the whole step."""
    import itertools

    import numpy as np

    from oracle import hotrg_oracle as o
    t0 = time.perf_counter()
    tp = o.to_paper_order(run.t, axis)
    nxt = o.next_axes(D, axis)
    legs = [o.choose_isometry(tp, j, CHI, nxt[j - 1]) for j in range(1, D)]
    t_env = time.perf_counter() - t0
    us = [leg.u for leg in legs]
    chi_c = tp.shape[2 * D - 2]
    nprimes = list(itertools.product(*[range(u.shape[1]) for u in us]))
    total_iters = chi_c * len(nprimes)
    t1 = time.perf_counter()
    that_mat = o.hat_matrix(tp)
    done = 0
    for c0p in range(chi_c):
        for npr in nprimes:
            o.new_tensor_slab(tp, us, c0p, npr, that_mat)
            done += 1
            if done >= sample_iters:
                break
        if done >= sample_iters:
            break
    t_con = time.perf_counter() - t1
    return t_env + t_con * total_iters / done, dict(env_eig_s=round(t_env, 3),
                                                   contraction_iters_timed=done,
                                                   contraction_iters_total=total_iters)


def fp64_form_leg(pkg, args, nsteps=2):
    """The plain FP64 form of the same workload on the GPU: the bond-growth steps, then
    `nsteps` steady steps timed with CUDA events (the first steady steps, where the Z2
    blocks are balanced: its cheapest steps), their ln Z/V against the oracle's reference,
    and the FP64 bottleneck rate as a fraction of the rate that bounds it (fp64_peak)."""
    import torch

    peak, peak_src = fp64_peak(pkg)
    stream = torch.cuda.current_stream()
    f = pkg.Hotrg(D, BETA, H, precision=pkg.PREC_FP64, z2=args.z2 == "on")
    axes = axes_for(GROWTH_STEPS + nsteps)
    for a in axes[:GROWTH_STEPS]:
        f.step(a, CHI)
    f.free_energy()
    pkg.hotrg_profile(f.ctx, 2)
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    done = 0.0
    torch.cuda.synchronize()
    ev0.record(stream)
    for a in axes[GROWTH_STEPS:]:
        f.step(a, CHI)
        done += pkg.hotrg_bottleneck_flops(f.ctx)[1]
    ev1.record(stream)
    torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1) / nsteps
    gemm_ms, gemm_n, _ = pkg.hotrg_step_times(f.ctx)
    lnz = f.free_energy()[0]
    f.close()
    golden = load_golden()
    last = GROWTH_STEPS + nsteps
    achieved = done / (gemm_ms["bottleneck"] / 1000.0) / 1e12 if gemm_ms["bottleneck"] > 0 else None
    return {"precision": "fp64", "steps_timed": f"{GROWTH_STEPS + 1}-{last}", "ms_per_step": ms,
            "steps_per_s": 1000.0 / ms,
            "rel_err_lnz_per_site_vs_oracle": abs(lnz - golden[last]) / abs(golden[last]) if last in golden else None,
            "bottleneck_flops_per_step": done / nsteps,
            "bottleneck_tflops": achieved, "fp64_bound_tflops": peak, "fp64_bound_source": peak_src,
            "frac_of_fp64_bound": achieved / peak if achieved else None,
            "note": "first steady steps (balanced Z2 blocks); later steps keep more even states and cost more"}


def cpu_baseline_leg():
    run = oracle_steady_tensor()
    est, info = oracle_step_sample(run, axes_for(GROWTH_STEPS + 1)[-1], 48)
    return {"value": 1.0 / est, "unit": "steps/s", "cores": os.cpu_count(), "kind": "oracle",
            "sample": (f"one steady-state step of {W['text']}: environments + Jacobi in full "
                       f"({info['env_eig_s']} s), {info['contraction_iters_timed']} of "
                       f"{info['contraction_iters_total']} (c'_0, n') contraction iterations, "
                       f"extrapolated to the whole step"),
            "extrapolated_s_per_step": est}


def reference_arm(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    run = oracle_steady_tensor()
    axes = axes_for(GROWTH_STEPS + args.warmup + args.steps)[GROWTH_STEPS:]
    ests = []
    for i, a in enumerate(axes):
        est, info = oracle_step_sample(run, a, 16)
        if i >= args.warmup:
            ests.append(est)
    mean = sum(ests) / len(ests)
    line = {"impl": "reference", "metric": METRIC, "value": 1.0 / mean, "unit": "steps/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1000.0 * mean, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": W["text"],
                       "sample": "each step: oracle environments + Jacobi in full and 16 "
                                 "contraction iterations, extrapolated"},
            "cpu_baseline": {"value": 1.0 / mean, "unit": "steps/s", "cores": os.cpu_count(),
                             "kind": "oracle", "sample": "16 contraction iterations per step, extrapolated"},
            "e2e": {"value": 1.0 / mean, "unit": "steps/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ---------------------------------------------------------------------------
# our arm
# ---------------------------------------------------------------------------

def batch_arm(args):
    """Batching form: 64 independent instances stepped together by hotrg_step_batch (one
    stream and one host worker per instance in flight), against the same instances
    stepped one after another.  Metric: instance-steps per second."""
    import torch

    import paper_2110_03607_gb300 as pkg

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    prec = prec_const(pkg, args.precision)
    inst = batch_instances()
    n = len(inst)
    streams = [torch.cuda.Stream() for _ in range(n)]
    ctxs = []
    for (beta, h, chi), st in zip(inst, streams):
        c = pkg.hotrg_init_ising(3, beta, h)
        pkg.hotrg_set_precision(c, prec)
        pkg.hotrg_set_z2(c, args.z2 == "on")
        pkg.hotrg_set_stream(c, st.cuda_stream)
        ctxs.append(c)
    chis = [x[2] for x in inst]
    nthreads = args.batch_threads
    total = GROWTH_STEPS + args.warmup + args.steps
    axes = [(FIRST_AXIS + s) % D for s in range(total)]
    for a in axes[: GROWTH_STEPS + args.warmup]:
        pkg.hotrg_step_batch(ctxs, [a] * n, chis, nthreads)
    timed = axes[GROWTH_STEPS + args.warmup:]
    graphs = None
    if args.graphs:
        # captured cycles: dense steps (parities dropped: no read-back), one uncaptured
        # cycle to place the buffers, then each instance's next 6-step cycle (lcm(2, 3))
        # recorded once; the timed region replays whole cycles
        cyc = 6
        for c in ctxs:
            pkg.hotrg_set_parity(c, None)
        ncyc = max(1, -(-len(timed) // cyc))
        ax_all = [(FIRST_AXIS + s) % D for s in range(GROWTH_STEPS + args.warmup + cyc * (ncyc + 1))]
        warm_cyc = ax_all[GROWTH_STEPS + args.warmup: GROWTH_STEPS + args.warmup + cyc]
        for a in warm_cyc:
            pkg.hotrg_step_batch(ctxs, [a] * n, chis, nthreads)
        cyc_axes = ax_all[GROWTH_STEPS + args.warmup + cyc: GROWTH_STEPS + args.warmup + 2 * cyc]
        graphs = [pkg.hotrg_graph_capture(c, cyc_axes, chi) for c, chi in zip(ctxs, chis)]
        timed = cyc_axes * ncyc
        axes = ax_all[: GROWTH_STEPS + args.warmup + cyc] + timed
    torch.cuda.synchronize()
    launches0 = pkg.hotrg_launch_count(ctxs[0])
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    flops = 0.0
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    if graphs is not None:
        for _ in range(len(timed) // 6):
            for c, gr in zip(ctxs, graphs):
                pkg.hotrg_graph_launch(c, gr)
    else:
        for a in timed:
            pkg.hotrg_step_batch(ctxs, [a] * n, chis, nthreads)
    torch.cuda.synchronize()
    elapsed_ms = (time.perf_counter() - t0) * 1000.0
    if graphs is not None:
        for gr in graphs:
            pkg.hotrg_graph_free(gr)
    if dist:
        dist.barrier()
    sampler.stop()
    launches = pkg.hotrg_launch_count(ctxs[0]) - launches0
    for c in ctxs:
        flops += pkg.hotrg_bottleneck_flops(c)[1]
    lnz = [pkg.hotrg_free_energy(c)[0] for c in ctxs]
    # the same instances, one after another (serial reference of the batching)
    torch.cuda.synchronize()
    t1 = time.perf_counter()
    for a in axes[GROWTH_STEPS + args.warmup: GROWTH_STEPS + args.warmup + 2]:
        for c, chi in zip(ctxs, chis):
            pkg.hotrg_step(c, a, chi)
        torch.cuda.synchronize()
    serial_ms = (time.perf_counter() - t1) * 1000.0 / 2
    # end to end: each instance's tensor from pinned host memory, one batch step, ln Z and
    # the tensors back
    e2e = None
    if not args.no_e2e:
        hosts, outs, dims, pars = [], [], [], []
        for c in ctxs:
            t = pkg.hotrg_tensor(c)
            p = torch.empty(t.size, dtype=torch.float64, pin_memory=True)
            p.numpy()[:] = t.reshape(-1)
            hosts.append(p)
            outs.append(torch.empty_like(p).pin_memory())
            dims.append(pkg.hotrg_bond_dims(c)[:3])
            pars.append(pkg.hotrg_leg_parity(c))
        a = axes[-1]
        torch.cuda.synchronize()
        t2 = time.perf_counter()
        h2d = d2h = 0
        for c, p, dm, par in zip(ctxs, hosts, dims, pars):
            pkg.hotrg_set_tensor(c, dm, p)
            h2d += p.numel() * 8
            if par is not None:
                pkg.hotrg_set_parity(c, par)
                h2d += 4 * len(par)
        pkg.hotrg_step_batch(ctxs, [a] * n, chis, nthreads)
        for c, o in zip(ctxs, outs):
            pkg.hotrg_free_energy(c)
            pkg.hotrg_tensor(c, o.numpy().reshape([x for x in pkg.hotrg_bond_dims(c)[:3] for _ in (0, 1)]))
            d2h += o.numel() * 8 + 16
        e2e_s = time.perf_counter() - t2
        e2e = {"value": n / e2e_s, "unit": "instance-steps/s", "h2d_bytes_per_step": h2d,
               "d2h_bytes_per_step": d2h, "steps": 1}
    clocks = sampler.summary()
    for c in ctxs:
        pkg.hotrg_free(c)
    elapsed_ms = max_over_ranks(elapsed_ms, dist, "cuda")
    K = len(timed)
    value = whole_job_rate(n * K, world, elapsed_ms)
    peaks, peak_src = load_peaks()
    peak = float(peaks.get("bf16_tflops_sustained", 1700.0))
    # flops: the performed bottleneck flops of one batch step (all instances' last step)
    achieved = flops / (elapsed_ms / K / 1000.0) / 1e12 if K else None
    if rank == 0:
        line = {
            "metric": "HOTRG instance-steps/s, batching form (64 independent 3D Ising instances)",
            "value": value, "unit": "instance-steps/s", "n_gpus": world, "steps": K,
            "warmup": args.warmup, "ms_per_step": elapsed_ms / K, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None,
            "dtype": PRECISIONS[args.precision][3],
            "data": "synthetic (Ising initial tensors from beta, h; no dataset)",
            "config": {"workload": W["text"] + f"; steps 1-{GROWTH_STEPS} (bond growth) untimed, "
                                   f"{args.warmup} warm-up steps, {K} timed batch steps",
                       "precision": args.precision,
                       "z2_blocks": args.z2 == "on" and not args.graphs,
                       "captured_graphs": "one 6-step cycle per instance, replayed" if args.graphs else None,
                       "host_workers": (1 if args.graphs else (nthreads if nthreads > 0 else "hardware threads")),
                       "l2": "not flushed: the 64 instances' tensors and operands (several GB) "
                             "exceed L2 together",
                       "parallelism": f"replicas x{world}" if world > 1 else "single GPU"},
            "serial_instance_steps_per_s": n / (serial_ms / 1000.0),
            "batching_speedup": value / world / (n / (serial_ms / 1000.0)),
            "ln_z_per_site_range": [min(lnz), max(lnz)],
            "roofline": {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                         "frac": achieved / peak if achieved else None, "traffic": None,
                         "peak_source": f"bf16_tflops_sustained of {peak_src}",
                         "note": "whole-job bottleneck GEMM flops (performed) per batch step / "
                                 "batch step wall time; kernels of different instances overlap"},
            "e2e": e2e,
            "gpu_launches": launches,
            "clocks": clocks,
            "cpu_baseline": None,
        }
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


def energy_arm(args):
    """Differentiation form: 3D Ising chi = 12 steps that carry d/d beta (dense contraction
    in the arithmetic of --precision) and end with the internal energy per site; the energy
    is checked against central differences (beta +- 1e-5, 1e-4) of FP64 runs over the same
    steps.  Metric: steps/s with the derivative carried."""
    import torch

    import paper_2110_03607_gb300 as pkg

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    stream = torch.cuda.current_stream()
    axes = axes_for(GROWTH_STEPS + args.warmup + args.steps)
    prec = prec_const(pkg, args.precision)
    g = pkg.Hotrg(D, BETA, H, precision=prec)
    pkg.hotrg_set_tangent(g.ctx, True)
    for a in axes[: GROWTH_STEPS + args.warmup]:
        g.step(a, CHI)
    pkg.hotrg_profile(g.ctx, 2)
    timed_axes = axes[GROWTH_STEPS + args.warmup:]
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    bn_done = 0.0
    launches0 = pkg.hotrg_launch_count(g.ctx)
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    ev0.record(stream)
    for a in timed_axes:
        g.step(a, CHI)
        bn_done += pkg.hotrg_bottleneck_flops(g.ctx)[1]
    ev1.record(stream)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    elapsed_ms = ev0.elapsed_time(ev1)
    launches = pkg.hotrg_launch_count(g.ctx) - launches0
    sampler.stop()
    clocks = sampler.summary()
    gemm_ms, gemm_n, _ = pkg.hotrg_step_times(g.ctx)
    dlnz, energy, degenerate = g.energy()
    lnz = g.free_energy()[0]
    g.close()
    elapsed_ms = max_over_ranks(elapsed_ms, dist, "cuda")
    K = len(timed_axes)
    value = whole_job_rate(K, world, elapsed_ms)

    # central differences of FP64 runs over the same steps (untimed), beta +- 1e-5 and 1e-4
    def ln_z_at(b):
        f = pkg.Hotrg(D, b, H, precision=pkg.PREC_FP64)
        for a in axes:
            f.step(a, CHI)
        v = f.free_energy()[0]
        f.close()
        return v

    fds = {db: (ln_z_at(BETA + db) - ln_z_at(BETA - db)) / (2 * db) for db in (1e-5, 1e-4)}
    fd = fds[1e-5]

    # roofline of the bottleneck region: per c'-slice one GEMM for C and two for
    # dC = T^ . dB^T + dT^ . B^T, each 2 R^2 Nc flops (algorithmic)
    n_regions = gemm_n["bottleneck"]
    region_ms = gemm_ms["bottleneck"] / max(1, n_regions)
    flops_per_region = 3.0 * bn_done / max(1, n_regions)
    achieved = flops_per_region / (region_ms / 1000.0) / 1e12 if region_ms > 0 else None
    if args.precision == "fp64":
        roof = {"bound": "alu", "achieved": achieved, "peak": 1.25, "unit": "TFLOP/s",
                "frac": achieved / 1.25 if achieved else None, "traffic": None,
                "peak_source": "nominal GB300 FP64 (no measured FP64 peak)"}
    else:
        peaks, peak_src = load_peaks()
        _, nterms, rate, _ = PRECISIONS[args.precision]
        peak = float(peaks.get("bf16_tflops_sustained", 1700.0)) * rate
        roof = {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                "frac": achieved / peak if achieved else None, "traffic": None,
                "peak_source": f"bf16_tflops_sustained of {peak_src}"
                               + ("" if rate == 1.0 else f" x {rate:.4f} (TF32 / BF16 nominal dense rate)"),
                "issued_tflops": achieved * nterms if achieved else None,
                "issued_frac": achieved * nterms / peak if achieved else None}
    roof["note"] = ("bottleneck region per c'-slice: three GEMMs of 2 R^2 Nc flops "
                    "(C, T^.dB^T, dT^.B^T) and one vector add")
    if rank == 0:
        line = {
            "metric": "3D-Ising chi=12 HOTRG steps/s carrying d/d beta (internal energy)",
            "value": value, "unit": "steps/s", "n_gpus": world, "steps": K, "warmup": args.warmup,
            "ms_per_step": elapsed_ms / K, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None,
            "dtype": PRECISIONS[args.precision][3],
            "data": "synthetic (Ising initial tensor and its beta-derivative from beta, h; no dataset)",
            "config": {"workload": W["text"] + f"; steps 1-{GROWTH_STEPS} (bond growth) untimed, "
                                   f"{args.warmup} warm-up steps, steps {GROWTH_STEPS + args.warmup + 1}-"
                                   f"{GROWTH_STEPS + args.warmup + K} timed",
                       "precision": args.precision, "z2_blocks": False,
                       "l2": "inputs larger than L2 (per-slice operands and their derivatives)",
                       "parallelism": f"replicas x{world}" if world > 1 else "single GPU"},
            "ln_z_per_site": lnz,
            "dlnz_dbeta_per_site": dlnz,
            "energy_per_site": energy,
            "energy_central_difference": -fd,
            "rel_err_energy_vs_central_difference": abs(dlnz - fd) / abs(fd),
            "rel_err_energy_vs_central_difference_by_step": {str(k): abs(dlnz - v) / abs(v)
                                                              for k, v in fds.items()},
            # the central difference errs by c db^2: one Richardson step removes that term
            "rel_err_energy_vs_richardson_extrapolated_difference":
                abs(dlnz - (fds[1e-5] - (fds[1e-4] - fds[1e-5]) / 99.0)) / abs(fd),
            "degenerate_pairs": degenerate,
            "roofline": roof,
            "e2e": None,
            "e2e_note": "inputs are beta and h only (the tensors are built on the device); "
                        "the end-to-end contract of the default workload does not apply",
            "gpu_launches": launches,
            "clocks": clocks,
            "cpu_baseline": None,
        }
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


def energy_scan_arm(args):
    """Differentiation form over a beta scan: 32 instances (beta uniform in [0.21, 0.23])
    carrying d/d beta, stepped together by hotrg_step_batch; the internal energy u(beta)
    after the last step and the specific heat c = -beta^2 du/dbeta by central differences
    on the grid; the middle instance's energy checked against central differences of FP64
    runs.  Metric: instance-steps/s."""
    import torch

    import paper_2110_03607_gb300 as pkg

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    prec = prec_const(pkg, args.precision)
    betas = [0.21 + 0.02 * i / 31.0 for i in range(32)]
    n = len(betas)
    streams = [torch.cuda.Stream() for _ in range(n)]
    ctxs = []
    for b, st in zip(betas, streams):
        c = pkg.hotrg_init_ising(D, b, H)
        pkg.hotrg_set_precision(c, prec)
        pkg.hotrg_set_stream(c, st.cuda_stream)
        pkg.hotrg_set_tangent(c, True)
        ctxs.append(c)
    total = GROWTH_STEPS + args.warmup + args.steps
    axes = axes_for(total)
    chis = [CHI] * n
    for a in axes[: GROWTH_STEPS + args.warmup]:
        pkg.hotrg_step_batch(ctxs, [a] * n, chis, args.batch_threads)
    torch.cuda.synchronize()
    timed = axes[GROWTH_STEPS + args.warmup:]
    launches0 = pkg.hotrg_launch_count(ctxs[0])
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for a in timed:
        pkg.hotrg_step_batch(ctxs, [a] * n, chis, args.batch_threads)
    torch.cuda.synchronize()
    elapsed_ms = (time.perf_counter() - t0) * 1000.0
    if dist:
        dist.barrier()
    sampler.stop()
    launches = pkg.hotrg_launch_count(ctxs[0]) - launches0
    res = [pkg.hotrg_energy(c) for c in ctxs]
    for c in ctxs:
        pkg.hotrg_free(c)
    u = [r[1] for r in res]
    deg = sum(r[2] for r in res)
    db_grid = betas[1] - betas[0]
    heat = {f"{betas[i]:.5f}": -betas[i] ** 2 * (u[i + 1] - u[i - 1]) / (2 * db_grid) for i in range(1, n - 1)}
    # the middle instance against central differences of FP64 runs (untimed)
    mid = n // 2

    def ln_z_at(b):
        f = pkg.Hotrg(D, b, H, precision=pkg.PREC_FP64)
        for a in axes:
            f.step(a, CHI)
        v = f.free_energy()[0]
        f.close()
        return v

    fds = {db: (ln_z_at(betas[mid] + db) - ln_z_at(betas[mid] - db)) / (2 * db) for db in (1e-5, 1e-4)}
    rich = fds[1e-5] - (fds[1e-4] - fds[1e-5]) / 99.0
    elapsed_ms = max_over_ranks(elapsed_ms, dist, "cuda")
    K = len(timed)
    value = whole_job_rate(n * K, world, elapsed_ms)
    if rank == 0:
        line = {
            "metric": "3D-Ising chi=12 HOTRG instance-steps/s carrying d/d beta, 32-beta scan",
            "value": value, "unit": "instance-steps/s", "n_gpus": world, "steps": K,
            "warmup": args.warmup, "ms_per_step": elapsed_ms / K, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None,
            "dtype": PRECISIONS[args.precision][3],
            "data": "synthetic (Ising initial tensors and their beta-derivatives from beta, h; no dataset)",
            "config": {"workload": W["text"] + f"; steps 1-{GROWTH_STEPS} (bond growth) untimed, "
                                   f"{args.warmup} warm-up steps, {K} timed batch steps",
                       "precision": args.precision, "instances": n,
                       "host_workers": args.batch_threads,
                       "l2": "not flushed: the 32 instances' operands (tens of GB) exceed L2 together",
                       "parallelism": f"replicas x{world}" if world > 1 else "single GPU"},
            "beta": betas,
            "energy_per_site": u,
            "specific_heat_per_site": heat,
            "degenerate_pairs": deg,
            "check_beta": betas[mid],
            "rel_err_energy_vs_central_difference": abs(-u[mid] - fds[1e-5]) / abs(fds[1e-5]),
            "rel_err_energy_vs_richardson_extrapolated_difference": abs(-u[mid] - rich) / abs(rich),
            "roofline": None,
            "roofline_note": "see the single-instance energy3d_chi12 line; kernels of different "
                             "instances overlap here",
            "e2e": None,
            "gpu_launches": launches,
            "clocks": sampler.summary(),
            "cpu_baseline": None,
        }
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


def shard_arm(args):
    """One run, its steps split by c'-slices over the ranks (NCCL collectives)."""
    import socket

    import torch
    import torch.distributed as dist

    import paper_2110_03607_gb300 as pkg
    from paper_2110_03607_gb300 import shard

    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world == 1 and "MASTER_PORT" not in os.environ:
        so = socket.socket()
        so.bind(("127.0.0.1", 0))
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        os.environ["MASTER_PORT"] = str(so.getsockname()[1])
        so.close()
        dist.init_process_group("nccl", rank=0, world_size=1)
    else:
        dist.init_process_group("nccl")
    rank = dist.get_rank()
    prec = prec_const(pkg, args.precision)
    stream = torch.cuda.current_stream()

    g = pkg.Hotrg(D, BETA, H, precision=prec, z2=args.z2 == "on")
    axes = axes_for(GROWTH_STEPS + args.warmup + args.steps)
    lnz_by_step = {}
    for i, a in enumerate(axes[: GROWTH_STEPS + args.warmup]):
        shard.step_sharded(g.ctx, a, CHI)
        lnz_by_step[i + 1] = g.free_energy()[0]
    timed_axes = axes[GROWTH_STEPS + args.warmup:]
    pkg.hotrg_profile(g.ctx, 2)
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    bn_done = 0.0
    launches0 = pkg.hotrg_launch_count(g.ctx)
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    lnz_timed = []
    dist.barrier()
    torch.cuda.synchronize()
    ev0.record(stream)
    for a in timed_axes:
        shard.step_sharded(g.ctx, a, CHI)            # synchronous: collectives between calls
        bn_done += pkg.hotrg_bottleneck_flops(g.ctx)[1]
        lnz_timed.append(g.free_energy()[0])         # 16-byte read-back after the gather
    ev1.record(stream)
    torch.cuda.synchronize()
    dist.barrier()
    elapsed_ms = max_over_ranks(ev0.elapsed_time(ev1), dist, "cuda")
    launches = pkg.hotrg_launch_count(g.ctx) - launches0
    sampler.stop()
    clocks = sampler.summary()
    gemm_ms, gemm_n, _ = pkg.hotrg_step_times(g.ctx)
    pkg.hotrg_profile(g.ctx, 0)
    K = len(timed_axes)
    for i, v in enumerate(lnz_timed):
        lnz_by_step[GROWTH_STEPS + args.warmup + i + 1] = v
    golden = load_golden()
    errs = {s: abs(lnz_by_step[s] - golden[s]) / abs(golden[s]) for s in lnz_by_step if s in golden}
    g.close()

    # roofline of this rank's bottleneck GEMM launches (its share of the c'-slices)
    peaks, peak_src = load_peaks()
    bn_launches = gemm_n.get("bottleneck", 0)
    bn_ms = gemm_ms.get("bottleneck", 0.0) / max(1, bn_launches)
    achieved = (bn_done / max(1, bn_launches)) / (bn_ms / 1000.0) / 1e12 if bn_ms > 0 else None
    _, nterms, rate, _ = PRECISIONS[args.precision]
    if args.precision == "fp64":
        peak, peak_src = fp64_peak(pkg)
        roof = {"bound": "tensor", "peak_source": peak_src}
    else:
        peak = float(peaks.get("bf16_tflops_sustained", 1700.0)) * rate
        roof = {"bound": "tensor", "peak_source": f"bf16_tflops_sustained of {peak_src}"
                + ("" if rate == 1.0 else f" x {rate:.4f} (TF32 / BF16 nominal dense rate)")}
    roof.update({"achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                 "frac": achieved / peak if achieved else None, "traffic": None,
                 "avg_launch_ms": bn_ms, "launches_per_step": bn_launches / K})

    if rank == 0:
        line = {
            "metric": METRIC, "value": K / (elapsed_ms / 1000.0), "unit": "steps/s", "n_gpus": world,
            "steps": K, "warmup": args.warmup, "ms_per_step": elapsed_ms / K, "higher_is_better": True,
            "scaling": "strong", "vs_baseline": None,
            "dtype": PRECISIONS[args.precision][3],
            "data": "synthetic (Ising initial tensor from beta, h; no dataset)",
            "config": {"workload": W["text"] + f"; steps 1-{GROWTH_STEPS} (bond growth) untimed, "
                                   f"{args.warmup} warm-up steps, "
                                   f"steps {GROWTH_STEPS + args.warmup + 1}-{GROWTH_STEPS + args.warmup + K} timed",
                       "precision": args.precision, "z2_blocks": args.z2 == "on",
                       "l2": "inputs larger than L2 (T 134 MB, per-slice operands GBs)",
                       "parallelism": f"c'-slice shard x{world} (NCCL all_reduce of the Grams, "
                                      f"all_gather of the new tensor's slices)"},
            "timing": "each timed step is the synchronous sharded step with its two collectives "
                      "and a 16-byte ln Z read-back",
            "rel_err_lnz_per_site_vs_oracle": max(errs.values()) if errs else None,
            "rel_err_steps_compared": len(errs),
            "roofline": roof,
            "e2e": None,
            "e2e_note": "the sharded step is host-synchronous already; the end-to-end number of the "
                        "one-process step is the default arm's",
            "gpu_launches": launches,
            "clocks": clocks,
            "cpu_baseline": None,
        }
        print(json.dumps(line), flush=True)
    dist.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=24)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--precision", default="bf16x6", choices=list(PRECISIONS))
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-fp64-form", action="store_true",
                    help="skip the two timed steps of the plain FP64 form")
    ap.add_argument("--workload", default="ising3d_chi16", choices=sorted(WORKLOADS))
    ap.add_argument("--autotune", action="store_true",
                    help="tune the chain stages' launch shapes on their first launch (hotrg_set_autotune)")
    ap.add_argument("--graphs", action="store_true",
                    help="batching workloads: replay captured 6-step cycles (dense steps) instead of "
                         "stepping through hotrg_step_batch")
    ap.add_argument("--batch-threads", type=int, default=16,
                    help="host workers of the batching form (batch3d_mixed)")
    ap.add_argument("--shard", action="store_true",
                    help="split each step of ONE run by c'-slices over the ranks (NCCL; strong scaling) "
                         "instead of running independent replicas")
    ap.add_argument("--z2", default="on", choices=["on", "off"],
                    help="Z2 block form of the contraction (on) or the paper's dense form (off)")
    args = ap.parse_args()
    select_workload(args.workload)
    if args.warmup < 3 and not args.workload.startswith("ising4d_chi1"):
        ap.error("--warmup must be >= 3")
    if args.impl == "reference":
        return reference_arm(args)
    if args.shard:
        if args.workload not in ("ising3d_chi16", "ising3d_chi20", "ising4d_chi6"):
            ap.error("--shard: the ising3d_chi16, ising3d_chi20 and ising4d_chi6 workloads")
        return shard_arm(args)
    if args.workload == "batch3d_mixed":
        return batch_arm(args)
    if args.workload == "energy3d_chi12":
        return energy_arm(args)
    if args.workload == "energy3d_chi12_scan":
        return energy_scan_arm(args)

    import torch

    import paper_2110_03607_gb300 as pkg

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    prec = prec_const(pkg, args.precision)
    stream = torch.cuda.current_stream()

    g = pkg.Hotrg(D, BETA, H, precision=prec, z2=args.z2 == "on")
    if args.autotune:
        pkg.hotrg_set_autotune(g.ctx, True)
    axes = axes_for(GROWTH_STEPS + args.warmup + args.steps)
    lnz_by_step = {}
    for i, a in enumerate(axes[: GROWTH_STEPS + args.warmup]):
        g.step(a, CHI)
        lnz_by_step[i + 1] = g.free_energy()[0]
    # timed region: no read-back inside; events only around the bottleneck GEMMs
    # (profile mode 2, summed over the timed steps and read once afterwards)
    pkg.hotrg_profile(g.ctx, 2)
    timed_axes = axes[GROWTH_STEPS + args.warmup:]

    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    bn_dense = bn_done = 0.0
    z2_steps = 0
    launches0 = pkg.hotrg_launch_count(g.ctx)
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    ev0.record(stream)
    for a in timed_axes:
        g.step(a, CHI)
        fd, fp, zb = pkg.hotrg_bottleneck_flops(g.ctx)   # host-side bookkeeping, no sync
        bn_dense += fd
        bn_done += fp
        z2_steps += int(zb)
    ev1.record(stream)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    elapsed_ms = ev0.elapsed_time(ev1)
    launches = pkg.hotrg_launch_count(g.ctx) - launches0
    sampler.stop()
    clocks = sampler.summary()
    elapsed_ms = max_over_ranks(elapsed_ms, dist, "cuda")
    K = len(timed_axes)
    value = whole_job_rate(K, world, elapsed_ms)
    gemm_ms, gemm_n, _ = pkg.hotrg_step_times(g.ctx)
    lnz_timed = g.free_energy()[0]
    pkg.hotrg_profile(g.ctx, 0)

    # ---- untimed replay of the same run (deterministic kernels: the same bits), with
    # per-step phase times and per-step ln Z / V for the accuracy check
    # (skipped for the paper-shape 4D workloads: a second run of a minutes-long step)
    phase_sum = {"bottleneck": gemm_ms["bottleneck"]}
    replay_same = None
    if not WORKLOAD.startswith("ising4d_chi1"):
        rp = pkg.Hotrg(D, BETA, H, precision=prec, z2=args.z2 == "on")
        if args.autotune:
            pkg.hotrg_set_autotune(rp.ctx, True)
        phase_sum = {}
        step_no = 0
        for i, a in enumerate(axes):
            if i == GROWTH_STEPS + args.warmup:
                pkg.hotrg_profile(rp.ctx, 1)
            rp.step(a, CHI)
            step_no += 1
            if i >= GROWTH_STEPS + args.warmup:
                ms, nl, f64 = pkg.hotrg_step_times(rp.ctx)
                for k, v in ms.items():
                    phase_sum[k] = phase_sum.get(k, 0.0) + v
            lnz_by_step[step_no] = rp.free_energy()[0]
        replay_same = lnz_by_step[step_no] == lnz_timed
        rp.close()
    launch_sum = {"bottleneck": gemm_n["bottleneck"]}
    phase_bn_ms = gemm_ms["bottleneck"]

    # ---- accuracy against the FP64 oracle's per-step ln Z / V (tests/golden)
    golden = load_golden()
    errs = {s: abs(lnz_by_step[s] - golden[s]) / abs(golden[s]) for s in lnz_by_step if s in golden}
    rel_err = max(errs.values()) if errs else None

    # ---- roofline of the bottleneck GEMM: algorithmic flops per launch (dense: one
    # launch of 2 R^2 Ns per c'-slice; Z2 blocks: two launches per c'-slice whose
    # flops, padding excluded, the library reports) / CUDA-event time per launch
    peaks, peak_src = load_peaks()
    bn_launches = launch_sum.get("bottleneck", 0)
    bn_ms = phase_bn_ms / max(1, bn_launches)
    flops_per_launch = bn_done / max(1, bn_launches)
    _, nterms, rate, _ = PRECISIONS[args.precision]
    achieved = flops_per_launch / (bn_ms / 1000.0) / 1e12 if bn_ms > 0 else None
    peak = float(peaks.get("bf16_tflops_sustained", 1700.0)) * (rate or 1.0)
    if args.precision == "fp64":
        f64_peak, f64_src = fp64_peak(pkg)
        roof = {"bound": "tensor", "achieved": achieved, "peak": f64_peak, "unit": "TFLOP/s",
                "frac": achieved / f64_peak if achieved else None, "traffic": None,
                "peak_source": f64_src}
    else:
        # DRAM bytes (read + write) of one Z2 block GEMM launch from the ncu capture in
        # profiles/tc_gemm_pair_kernel_ising3d_chi16_bf16x6.md (the block shape of the first
        # steady steps: M = K = 2048, N = 32768); only for that workload and form
        traffic = (0.587e9 + 0.246e9) if (WORKLOAD == "ising3d_chi16" and args.precision == "bf16x6"
                                          and args.z2 == "on") else None
        roof = {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                "frac": achieved / peak if achieved else None, "traffic": traffic,
                "traffic_note": "bytes per launch at the step-4..7 launch shape (M=K=2048, N=32768); "
                                "later steps have unequal blocks" if traffic else None,
                "peak_source": f"bf16_tflops_sustained of {peak_src}"
                               + ("" if rate == 1.0 else f" x {rate:.4f} (TF32 / BF16 nominal dense rate)"),
                "issued_tflops": achieved * nterms if achieved else None,
                "issued_frac": achieved * nterms / peak if achieved else None,
                "algorithmic_flops_per_launch": flops_per_launch,
                "avg_launch_ms": bn_ms,
                "launches_per_step": bn_launches / K,
                "dense_equivalent_tflops": (bn_dense / K) / (phase_bn_ms / K / 1000.0)
                / 1e12 if bn_launches else None}

    # ---- end to end through the public API with host buffers: a fresh run of the same
    # steps, the timed ones each taking its input tensor from pinned host memory and
    # returning ln Z and the new tensor to the host
    e2e = None
    if not args.no_e2e:
        g.close()
        ee = pkg.Hotrg(D, BETA, H, precision=prec, z2=args.z2 == "on")
        for a in axes[: GROWTH_STEPS + args.warmup]:
            ee.step(a, CHI)
        t_host = pkg.hotrg_tensor(ee.ctx)
        pinned = torch.empty(t_host.size, dtype=torch.float64, pin_memory=True)
        pinned.numpy()[:] = t_host.reshape(-1)
        out = torch.empty_like(pinned).pin_memory()
        chis = pkg.hotrg_bond_dims(ee.ctx)[:D]
        parity = pkg.hotrg_leg_parity(ee.ctx)
        e2e_axes = timed_axes
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        h2d = d2h = 0
        for a in e2e_axes:
            pkg.hotrg_set_tensor(ee.ctx, chis, pinned)     # host -> device
            h2d += pinned.numel() * 8
            if parity is not None:                         # declared leg parities (Z2)
                pkg.hotrg_set_parity(ee.ctx, parity)
                h2d += 4 * len(parity)
            ee.step(a, CHI)
            parity = pkg.hotrg_leg_parity(ee.ctx)
            pkg.hotrg_free_energy(ee.ctx)                   # 16-byte read-back
            pkg.hotrg_tensor(ee.ctx, out.numpy().reshape([c for c in chis for _ in (0, 1)]))
            d2h += out.numel() * 8 + 16
            pinned, out = out, pinned
        dt = time.perf_counter() - t0
        e2e = {"value": len(e2e_axes) / dt, "unit": "steps/s",
               "h2d_bytes_per_step": h2d // len(e2e_axes), "d2h_bytes_per_step": d2h // len(e2e_axes),
               "steps": len(e2e_axes), "same_steps_as_value": True}
        g = ee
    g.close()

    # ---- the plain FP64 form of the same workload, for the metric's comparison
    fp64_form = None
    if args.precision != "fp64" and not args.no_fp64_form and WORKLOAD == "ising3d_chi16":
        fp64_form = fp64_form_leg(pkg, args)
        fp64_form["split_form_speedup"] = (value / world) / fp64_form["steps_per_s"]

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline and WORKLOAD in ("ising3d_chi16", "ising4d_chi6"):
        cpu = cpu_baseline_leg()

    if rank == 0:
        mean_phase = {k: round(v / K, 3) for k, v in phase_sum.items()}
        line = {
            "metric": METRIC, "value": value, "unit": "steps/s", "n_gpus": world, "steps": K,
            "warmup": args.warmup, "ms_per_step": elapsed_ms / K, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None,
            "dtype": PRECISIONS[args.precision][3],
            "data": "synthetic (Ising initial tensor from beta, h; no dataset)",
            "config": {"workload": W["text"] + f"; steps 1-{GROWTH_STEPS} (bond growth) untimed, "
                                   f"{args.warmup} warm-up steps, "
                                   f"steps {GROWTH_STEPS + args.warmup + 1}-{GROWTH_STEPS + args.warmup + K} timed",
                       "precision": args.precision,
                       "z2_blocks": args.z2 == "on",
                       "autotune": bool(args.autotune),
                       "z2_steps_timed": z2_steps,
                       "bottleneck_flops_per_step": {"dense": bn_dense / K, "performed": bn_done / K},
                       "l2": "inputs larger than L2 (T 134 MB, per-slice operands GBs)",
                       "parallelism": f"replicas x{world}" if world > 1 else "single GPU"},
            "timing": "timed steps run back to back without read-back; per-step ln Z / V and phase "
                      "times come from an untimed replay of the same run",
            "replay_matches_timed_run": replay_same,
            "rel_err_lnz_per_site_vs_oracle": rel_err,
            "rel_err_steps_compared": len(errs),
            "rel_err_by_step": {str(k): v for k, v in sorted(errs.items())},
            "phases_ms_per_step": mean_phase,
            "roofline": roof,
            "fp64_form": fp64_form,
            "e2e": e2e,
            "gpu_launches": launches,
            "clocks": clocks,
            "cpu_baseline": cpu,
        }
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
