#!/usr/bin/env python
"""Benchmark of the DP-SGD ghost-clipping hot path on B200.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference] [--workload cfg3]
    python bench.py --case gemm --reps 3          # one entry point on a small case (for profilers)

A step is one pass of the whole path over one synthetic batch: per-example norms of every
block linear layer, the LM head and the embedding (plus the tied cross term / position table
where the workload has them), clip factors, the clipped sum of every parameter tensor and its
Gaussian noise.  Prints ONE JSON line (rank 0).  The default workload is the GPT-2-small shape
(cfg3); at one GPU the line also carries a `sweep` over the other configurations, the
ghost-vs-direct timing per layer shape (`norm_modes`) and the tied path's extra cost.
`--impl reference` times the float64 CPU oracle instead (a reported baseline, not a target).
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time
import types

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "dp_sgd_examples_per_sec"
UNIT = "examples/s"

# DRAM bytes of the clipped-sum GEMM (dram__bytes_read.sum + dram__bytes_write.sum, one ncu capture
# of a three-wave, head-like launch each of gemm_gta_big_kernel and gemm_gta_kernel, 0.97 for both) divided
# by that launch's algorithmic bytes (inputs read once + fp32 outputs written once).  `roofline.traffic` of a workload is this ratio times
# the algorithmic bytes of its own grouped launch: the kernel reads every operand tile from DRAM
# once whatever the layer list, so traffic grows in proportion to the bytes.
GEMM_DRAM_OVER_ALGORITHMIC = 0.97


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return {"hbm_gbs": p["hbm_gbs"], "bf16_tflops": p["bf16_tflops"],
                "bf16_tflops_sustained": p.get("bf16_tflops_sustained", p["bf16_tflops"]),
                "source": "measured"}
    return {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0,
            "source": "fallback"}


def gemm_kernel_name(ds, reserved_sms):
    """The kernel behind the grouped clipped sums: items of two 256 x 256 tiles where every CTA pair gets two tiles."""
    import torch
    sms = torch.cuda.get_device_properties(ds.sq.device).multi_processor_count - reserved_sms
    layers = ds.linears + ([ds.lm] if ds.lm else [])
    tiles = sum(-(-l.p // 256) * -(-l.d // 256) for l in layers)
    return "gemm_gta_big_kernel" if tiles >= 2 * (sms // 2) else "gemm_gta_kernel<scale, pair>"


# ------------------------------------------------------------------------------- clocks
class ClockSampler:
    """Samples SM clock, power and throttle reasons with nvidia-smi while timed regions run."""
    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._pump, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _pump(self):
        for line in self.proc.stdout:
            self.lines.append((time.time(), line.strip()))

    def window(self, t0: float, t1: float):
        """Summary of the samples taken between two wall-clock times."""
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        sm, mx, reasons, power = [], [], set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ts, line in list(self.lines):
            if ts < t0 - 0.05 or ts > t1 + 0.15:
                continue
            f = [x.strip() for x in line.split(",")]
            try:
                sm.append(float(f[0])); mx.append(float(f[1])); power.append(float(f[2]))
            except (ValueError, IndexError):
                continue
            for n, v in zip(names, f[3:7]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None,
                "power_w_max": max(power) if power else None,
                "samples": len(sm), "reasons": sorted(reasons)}

    def stop(self):
        if self.proc is not None:
            time.sleep(0.15)
            self.proc.terminate()


def choose_tensor_peak(peaks, region_s, clocks):
    """Which measured bf16 peak a tensor-bound kernel of this run is compared with: the sustained
    (power-capped) figure only when the timed region itself was sustained -- at least a second
    long AND the sampler saw the power cap -- otherwise the burst figure."""
    capped = bool(clocks) and "sw_power_cap" in (clocks.get("reasons") or [])
    if region_s >= 1.0 and capped:
        return peaks["bf16_tflops_sustained"], "sustained", (
            "timed region %.2f s with sw_power_cap active (median SM clock %s MHz): sustained peak"
            % (region_s, clocks.get("sm_mhz")))
    why = []
    if region_s < 1.0:
        why.append("timed region only %.3f s" % region_s)
    if not capped:
        why.append("power cap not reached (median SM clock %s MHz)" % (clocks or {}).get("sm_mhz"))
    return peaks["bf16_tflops"], "burst", "; ".join(why) + ": burst peak"


# --------------------------------------------------------------------- algorithmic work
def work_counts(w):
    """Algorithmic bytes / flops of one step (per-unit figures times the units of the batch)."""
    B, T = w.B, w.T
    es = 2 if w.dtype == "bf16" else 4
    lin = [(l.d, l.p) for l in w.linears] + ([(w.lm.d, w.lm.p)] if w.lm else [])
    norm_bytes = sum(es * B * T * (d + p) for d, p in lin)
    gram_flops = sum(B * T * (T + 1) * (d + p) for d, p in lin)
    acc_flops = sum(2 * B * T * d * p for d, p in lin)
    acc_bytes = sum(es * B * T * (d + p) + 4 * d * p for d, p in lin)
    n_params = sum(d * p for d, p in lin) + w.V * w.d_model * (0 if (w.tied and w.lm) else 1)
    if w.positions:
        n_params += 1024 * w.d_model
    embed_bytes = es * B * T * w.d_model + 4 * B * T
    return dict(norm_bytes=norm_bytes, gram_flops=gram_flops, acc_flops=acc_flops,
                acc_bytes=acc_bytes, noise_bytes=8 * n_params, n_params=n_params,
                embed_bytes=embed_bytes)


def shape_of(ds, name):
    """The fields work_counts needs, from a device step."""
    return types.SimpleNamespace(
        name=name, dtype="bf16" if ds.G_emb.dtype.itemsize == 2 else "f32", B=ds.B, T=ds.T, V=ds.V,
        d_model=ds.d_model, tied=ds.tied, positions=ds.positions,
        linears=[types.SimpleNamespace(d=l.d, p=l.p) for l in ds.linears],
        lm=types.SimpleNamespace(d=ds.lm.d, p=ds.lm.p) if ds.lm else None)


def make_workload(name, seed=0, B=None, T=None, full_model=False):
    from paper_2609_40335_b200 import workloads
    over = {"full_model": True} if full_model else {}
    if B:
        over["B"] = B
    if T:
        over["T"] = T
    return workloads.named_workload(name, seed=seed, **over)


# ------------------------------------------------------------------------ reference arm
def oracle_layers_step(w, n_layers):
    """Only the first n linear layers of example 0 through the oracle (norm, clip factor, clipped
    sum): the short step of a reference run with many steps.  Returns seconds."""
    from oracle import dp_oracle as O
    sl = slice(0, 1)
    t0 = time.perf_counter()
    for l in w.linears[:n_layers]:
        A, G = l.A.widened_rows(sl), l.G.widened_rows(sl)
        sq = O.linear_sq_norms(A, G)
        _, R = O.clip_factors(sq, w.C)
        O.clipped_sum_linear(A, G, R)
    return time.perf_counter() - t0


def oracle_sample_step(w, n_examples):
    """The oracle, as it stands, on the first n examples of the workload (norms, clip factors,
    clipped sums of every parameter tensor).  Returns seconds."""
    from oracle import dp_oracle as O
    sl = slice(0, n_examples)
    t0 = time.perf_counter()
    lin = [(l.A.widened_rows(sl), l.G.widened_rows(sl)) for l in w.linears]
    lm = (w.lm.A.widened_rows(sl), w.lm.G.widened_rows(sl)) if w.lm else None
    O.dp_step(lin, w.ids[sl], w.G_emb.widened_rows(sl), w.V, w.C, lm=lm, tied=w.tied,
              positions=w.positions)
    return time.perf_counter() - t0


def oracle_noise_seconds(n):
    from oracle import noise_oracle as NO
    import numpy as np
    t0 = time.perf_counter()
    NO.add_noise(np.zeros(n), 1.0, 1.0, 1.0, 0, 0, 0)
    return time.perf_counter() - t0


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    cores = len(os.sched_getaffinity(0))
    w = make_workload(args.workload, B=args.B, T=args.T)
    # A step is one example through every layer when K such steps fit in ~2.5 minutes.  Otherwise a
    # step is the first few linear layers of one example, and its time is scaled to a whole example
    # by the ratio (whole example : those layers) measured once before the timed steps.
    oracle_sample_step(w, 1)                      # cold caches, lazy imports
    t_full = oracle_sample_step(w, 1)
    n_layers, ratio = None, 1.0
    if args.steps * t_full > 150.0:
        n_layers = 1
        t_sub = oracle_layers_step(w, 1)
        while n_layers < len(w.linears) and args.steps * t_sub * (n_layers + 1) / n_layers <= 150.0:
            n_layers += 1
            t_sub = oracle_layers_step(w, n_layers)
        ratio = t_full / t_sub
    for _ in range(max(0, args.warmup - 2)):
        oracle_sample_step(w, 1) if n_layers is None else oracle_layers_step(w, n_layers)
    ts = [(oracle_sample_step(w, 1) if n_layers is None else oracle_layers_step(w, n_layers))
          for _ in range(args.steps)]
    per = sum(ts) / len(ts) * ratio
    val = 1.0 / per
    sample = (f"each step = the float64 oracle on 1 of the {w.B} examples of {w.name} ("
              + ("all layers, norms + clip factors + clipped sums" if n_layers is None else
                 f"the first {n_layers} of {len(w.linears)} linear layers; step time scaled by "
                 f"{ratio:.1f}, the measured ratio of a whole example to those layers")
              + "; noise not included)")
    line = {"impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": per * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": w.name, "B_per_gpu": w.B, "T": w.T},
            "cpu_baseline": {"value": val, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)


# ----------------------------------------------------------------- device-side measurements
def _ev():
    import torch
    return torch.cuda.Event(enable_timing=True)


def time_graph(fn, reps, rounds=3):
    """Best-of-`rounds` device time of one call of fn, from a CUDA graph holding `reps` calls
    (the host's per-call work -- tensor-map encodes, argument checks -- stays out of the figure)."""
    import torch
    fn()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(reps):
            fn()
    g.replay()
    torch.cuda.synchronize()
    best = float("inf")
    a, b = _ev(), _ev()
    for _ in range(rounds):
        a.record()
        g.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / reps)
    return best


def graph_phase_times(P, ds, seed, first_step, replays, batches=5):
    """Per-phase and GEMM durations inside back-to-back replays of the captured step: a second
    capture of the same step with external event nodes is replayed in `batches` runs of
    replays/batches replays each (no synchronize inside a run, so the clock and power state are
    those of the timed region) and the events of each run's LAST replay are read."""
    import torch
    sgt = P.StepGraph(ds, seed=seed, first_step=first_step, timing=True)
    per = max(1, replays // batches)
    det = []
    for _ in range(batches):
        for _ in range(per):
            sgt.replay()
        torch.cuda.synchronize()
        det.append(sgt.phase_ms())
    med = lambda k: statistics.median(d[k] for d in det)
    return {"norms": med("norms"), "clip_accumulate": med("clip_accumulate"), "gemm": med("gemm"),
            "step_with_event_nodes": med("step"), "samples": len(det), "replays_per_sample": per}


def ghost_norm_alone(dp, ds, peaks, peak_tf, counts):
    """The linear-layer norm call alone (five calls in one graph, each with its reduce)."""
    import torch
    lin_layers = ds.linears + ([ds.lm] if ds.lm else [])
    ms = time_graph(lambda: dp.dp_ghost_norms(lin_layers, ds.B, ds.T, ds.sq, ws=ds.ws,
                                              dev_status=ds.dev_status), reps=5)
    t_hbm = counts["norm_bytes"] / (peaks["hbm_gbs"] * 1e9)
    t_tc = counts["gram_flops"] / (peak_tf * 1e12)
    return {"kernel": "ghost_norm_pair_kernel" if ds.T > 128 else "ghost_norm_tc_kernel",
            "bound": "hbm" if t_hbm >= t_tc else "tensor", "ms": ms,
            "achieved_GBs": counts["norm_bytes"] / (ms * 1e-3) / 1e9,
            "achieved_TFLOPs": counts["gram_flops"] / (ms * 1e-3) / 1e12,
            "peak_GBs": peaks["hbm_gbs"], "peak_TFLOPs": peak_tf,
            "frac": max(t_hbm, t_tc) * 1e3 / ms,
            "note": "frac = max(algorithmic bytes / HBM peak, symmetric-Gram flops / tensor peak) / measured"}


def measure_cell(P, dp, name, B, T, d_model, n_blocks, tied, positions, sigma, peaks, sampler, seed,
                 warmup=3, replays=10):
    """One configuration with inputs drawn on the device: replays of the captured step graph."""
    import torch
    dev = torch.cuda.current_device()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    ds = P.synthesize_on_device(name, B, T, d_model, n_blocks, tied=tied, positions=positions,
                                sigma=sigma, seed=seed)
    # footprint of the step itself: resident inputs + outputs + workspaces (the staging buffers of
    # the input synthesis are gone by now)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    torch.cuda.reset_peak_memory_stats(dev)
    counts = work_counts(shape_of(ds, name))
    sg = P.StepGraph(ds, seed=seed, first_step=0)
    for _ in range(warmup):
        sg.replay()
    torch.cuda.synchronize()
    a, b = _ev(), _ev()
    t0 = time.time()
    a.record()
    for _ in range(replays):
        sg.replay()
    b.record()
    torch.cuda.synchronize()
    t1 = time.time()
    assert int(ds.dev_status.item()) == 0, "device status flagged a problem in %s B=%d T=%d" % (name, B, T)
    ms = a.elapsed_time(b) / replays
    clocks = sampler.window(t0, t1) if sampler else None
    peak_tf, which, why = choose_tensor_peak(peaks, (t1 - t0), clocks)
    ph = graph_phase_times(P, ds, seed, warmup + replays, replays, batches=3)
    gemm_tf = counts["acc_flops"] / (ph["gemm"] * 1e-3) / 1e12
    ghost = ghost_norm_alone(dp, ds, peaks, peak_tf, counts)
    cell = {"workload": name, "B": B, "T": T, "blocks": n_blocks, "d_model": d_model, "tied": tied,
            "positions": positions, "replays": replays, "ms_per_step": ms,
            "examples_per_s": B / (ms * 1e-3), "norms_ms": ph["norms"],
            "clip_accumulate_ms": ph["clip_accumulate"], "norm_plus_clip_ms": ph["norms"] + ph["clip_accumulate"],
            "gemm": {"ms": ph["gemm"], "achieved_TFLOPs": gemm_tf, "peak_TFLOPs": peak_tf,
                     "peak": which, "frac": gemm_tf / peak_tf},
            "ghost_norm": {k: ghost[k] for k in ("kernel", "bound", "ms", "achieved_GBs",
                                                   "achieved_TFLOPs", "frac")},
            "input_bytes": int(ds.input_bytes()),
            "max_memory_allocated_bytes": int(torch.cuda.max_memory_allocated(dev)),
            "clocks": clocks}
    return cell, ds


def cross_term_alone(dp, ds):
    """The tied cross-term call alone (five calls in one graph), in microseconds."""
    import torch
    sq = torch.zeros_like(ds.sq)
    ms = time_graph(lambda: dp.dp_tied_cross_term(ds.ids, ds.G_emb, ds.lm.A, ds.lm.G, ds.V, sq=sq,
                                                  cross=ds.cross, d=ds.d_model, ws=ds.ws,
                                                  dev_status=ds.dev_status), reps=5)
    return ms * 1e3


def norm_modes(dp, ds, peaks):
    """GHOST against DIRECT per distinct layer shape of this workload (the per-layer switch):
    device time of one dp_ghost_norms call on that one layer in each forced mode, and what the
    AUTO rule (DIRECT iff T^2 > d p) picks."""
    import torch
    seen, rows = set(), []
    for l in ds.linears + ([ds.lm] if ds.lm else []):
        if (l.d, l.p) in seen:
            continue
        seen.add((l.d, l.p))
        sq = torch.zeros_like(ds.sq)
        row = {"d": l.d, "p": l.p, "T": ds.T, "B": ds.B}
        for label, mode in (("ghost_ms", dp.DP_NORM_GHOST), ("direct_ms", dp.DP_NORM_DIRECT)):
            one = dp.Linear(l.A, l.G, d=l.d, p=l.p, mode=mode)
            ws = torch.empty(max(256, dp.dp_ghost_norms_ws_bytes([one], ds.B, ds.T)), dtype=torch.uint8,
                             device=sq.device)
            row[label] = time_graph(lambda: dp.dp_ghost_norms([one], ds.B, ds.T, sq, ws=ws,
                                                               dev_status=ds.dev_status), reps=3)
        auto = dp.Linear(l.A, l.G, d=l.d, p=l.p, mode=dp.DP_NORM_AUTO)
        used = dp.dp_ghost_norms([auto], ds.B, ds.T, sq, dev_status=ds.dev_status)
        row["auto_chose"] = "direct" if used[0] == dp.DP_NORM_DIRECT else "ghost"
        row["direct_TFLOPs"] = 2.0 * ds.B * ds.T * l.d * l.p / (row["direct_ms"] * 1e-3) / 1e12
        row["ghost_GBs"] = 2.0 * ds.B * ds.T * (l.d + l.p) / (row["ghost_ms"] * 1e-3) / 1e9
        rows.append(row)
    torch.cuda.synchronize()
    return rows


SWEEP_CELLS = [
    # name, B, T, d_model, blocks, tied, positions, sigma
    ("cfg2", 32, 128, 768, 6, False, False, 0.8),
    ("cfg4", 32, 128, 768, 12, True, False, 0.8),
    ("cfg5", 16, 128, 1024, 24, False, False, 1.0),
    ("cfg5", 64, 128, 1024, 24, False, False, 1.0),
    ("cfg5", 256, 128, 1024, 24, False, False, 1.0),
    ("cfg5", 16, 512, 1024, 24, False, False, 1.0),
    ("cfg5", 64, 512, 1024, 24, False, False, 1.0),
    ("cfg5", 256, 512, 1024, 24, False, False, 1.0),
]


def run_sweep(P, dp, peaks, sampler, seed):
    """The other configurations, a few graph replays each, inputs drawn on the device.  Under cfg4
    (tied) also: the cross-term kernel alone, the same shape untied, peak memory of both."""
    import torch
    out, tied_cost = [], None
    for (name, B, T, dm, nb, tied, pos, sigma) in SWEEP_CELLS:
        cell, ds = measure_cell(P, dp, name, B, T, dm, nb, tied, pos, sigma, peaks, sampler, seed)
        if tied:
            cross_us = cross_term_alone(dp, ds)
            del ds
            untied, ds2 = measure_cell(P, dp, name + "-untied", B, T, dm, nb, False, pos, sigma, peaks,
                                       sampler, seed)
            del ds2
            tied_cost = {
                "shape": "B=%d T=%d, %d blocks, d=%d, V=50257" % (B, T, nb, dm),
                "cross_term_kernel_us": cross_us,
                "tied_ms_per_step": cell["ms_per_step"], "untied_same_shape_ms_per_step": untied["ms_per_step"],
                "step_delta_ms": cell["ms_per_step"] - untied["ms_per_step"],
                "tied_norms_ms": cell["norms_ms"], "untied_norms_ms": untied["norms_ms"],
                "tied_max_memory_allocated_bytes": cell["max_memory_allocated_bytes"],
                "untied_max_memory_allocated_bytes": untied["max_memory_allocated_bytes"],
                "note": ("tied: one shared 50257 x d matrix receives the head GEMM and the token scatter; "
                         "untied holds two.  The cross term is 2<g_in, g_out> per example through the "
                         "T x T pair expansion (no V x d matrix is formed)")}
        else:
            del ds
        out.append(cell)
        torch.cuda.empty_cache()
    return out, tied_cost


# ------------------------------------------------------------------------------ our arm
def run_ours(args):
    import torch
    import torch.distributed as dist

    from paper_2609_40335_b200 import binding as dp
    from paper_2609_40335_b200 import parallel
    from paper_2609_40335_b200 import pipeline as P

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the product path has no CPU fallback")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    reserve = args.reserve_sms
    if world > 1:
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        # The collectives run beside persistent kernels that take every SM they are given (and all
        # of its shared memory): cap the collectives' CTAs and leave them that many SMs.  With no
        # free SM a collective waits for the end of the running launch and then delays part of the
        # next one by a whole wave (measured on one GPU with a stand-in kernel: +36 % on the
        # clipped-sum phase, against 3 % for 16 SMs set aside).
        os.environ.setdefault("NCCL_MAX_CTAS", "16")
        if reserve is None:
            try:
                reserve = max(0, int(os.environ["NCCL_MAX_CTAS"]))
            except ValueError:
                reserve = 16
        dist.init_process_group("nccl", device_id=dev)
    dp.load()
    reserve = int(reserve or 0)
    dp.dp_set_reserved_sms(reserve)
    peaks = measured_peaks()

    # every rank holds its own batch of the same shape (weak scaling over examples)
    if args.device_inputs:
        assert args.workload == "cfg5", "--device-inputs is for the GPT-2-medium sweep"
        B_, T_ = args.B or 16, args.T or 128
        ds = P.synthesize_on_device("cfg5", B_, T_, 1024, 24, seed=rank, device=dev)
        w = shape_of(ds, "cfg5")
    else:
        w = make_workload(args.workload, seed=rank, B=args.B, T=args.T, full_model=args.full_model)
        ds = P.upload(w, dev)
    counts = work_counts(w)
    stream = torch.cuda.current_stream()

    fused = (world == 1) and not args.unfused and not args.bucketed     # noise inside the clipped-sum kernels
    exchange = None
    if (world > 1 or args.bucketed) and args.exchange == "reduce_scatter":
        # bucketed reduce-scatter on a communication stream; each rank noises the slices it owns
        step_box = [0]
        exchange = parallel.BucketedExchange(
            ds.outs, lambda t, first, tid, st: dp.dp_add_noise_slice(
                t, first, ds.sigma, ds.C, 1.0, args.seed, tid, step_box[0], stream=st),
            gather=args.gather)

    def step(k, ev=None):
        ge = (ev[4], ev[5]) if ev else None
        if ev: ev[0].record(stream)
        if fused and args.prefill:
            filled = P.prefill_all_noise(ds, args.seed, k)           # side stream, overlaps the norms
        if fused and not args.prefill:
            filled = P.overlapped_norms(ds, args.seed, k)            # noise fill beside the norm kernel
        else:
            P.norms_phase(ds)
        if ev: ev[1].record(stream)
        if fused and args.prefill:
            P.clip_onto_noise(ds, filled)
            if ev: ev[2].record(stream)
        elif fused:
            P.clip_after_prefill(ds, args.seed, k, filled, gemm_events=ge)
            if ev: ev[2].record(stream)
        elif exchange is not None:
            # N > 1 (default): the clipped sums leave bucket by bucket while the next bucket computes
            step_box[0] = k
            exchange.begin_step()
            P.clip_phase_bucketed(ds, exchange)
            if ev: ev[2].record(stream)
            exchange.finish()
        else:
            P.clip_phase(ds, gemm_events=ge)
            if ev: ev[2].record(stream)
            if world > 1:
                parallel.reduce_clipped_sums(ds.outs)
            P.noise_phase(ds, seed=args.seed, step=k)
        if ev: ev[3].record(stream)

    # default at N = 1: the whole step captured once as a CUDA graph and replayed (the noise step
    # advances on the device); --eager issues the same calls one by one instead
    use_graph = (world == 1) and fused and not args.prefill and not args.eager
    sg = None
    graph_note = None
    if use_graph:
        try:
            sg = P.StepGraph(ds, seed=args.seed, first_step=0)
        except Exception as e:           # capture refused on this stack: time the same calls eagerly
            torch.cuda.synchronize()
            dp.dp_noise_step_device(None)
            use_graph = False
            graph_note = "graph capture failed (%s: %s); the step was issued call by call" % (
                type(e).__name__, str(e).splitlines()[0][:120] if str(e) else "")
    eager_step = step
    if use_graph:
        def step(k, ev=None):          # noqa: F811  (replaces the eager step for every later use)
            sg.replay()

    for k in range(args.warmup):
        step(k)
    torch.cuda.synchronize()
    assert int(ds.dev_status.item()) == 0, "device status %#x flagged a problem during warm-up" % int(ds.dev_status.item())

    sampler = ClockSampler(local) if rank == 0 else None
    if sampler:
        sampler.start()
        time.sleep(0.25)
    evs = [[_ev() for _ in range(6)] for _ in range(args.steps)] if not use_graph else None
    e0, e1 = _ev(), _ev()
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    launches0 = dp.dp_kernel_launches()
    t_wall0 = time.time()
    e0.record(stream)
    for k in range(args.steps):
        step(args.warmup + k, evs[k] if evs else None)
    e1.record(stream)
    torch.cuda.synchronize()
    t_wall1 = time.time()
    if world > 1:
        dist.barrier()
    launches = dp.dp_kernel_launches() - launches0
    if use_graph:
        launches = sg.kernels_per_replay * args.steps      # replays do not pass through the library
    clocks = sampler.window(t_wall0, t_wall1) if sampler else None
    ms_total = e0.elapsed_time(e1)
    if world > 1:
        t = torch.tensor([ms_total], device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        ms_total = float(t.item())
    assert int(ds.dev_status.item()) == 0, "device status flagged a problem in the timed region"
    ms_step = ms_total / args.steps
    value = world * w.B / (ms_step * 1e-3)
    peak_tf, peak_kind, peak_why = choose_tensor_peak(peaks, ms_total * 1e-3, clocks)

    graph_detail = None
    if use_graph:
        ph = graph_phase_times(P, ds, args.seed, args.warmup + args.steps, args.steps)
        ms_norm, ms_clip, ms_noise, gemm_ms_avg = ph["norms"], ph["clip_accumulate"], 0.0, ph["gemm"]
        graph_detail = {"how": "phases and the GEMM are timed by external CUDA events inside a second "
                               "capture of the same step (the event nodes cost tens of microseconds per "
                               "step, so the timed region replays a capture without them): %d runs of "
                               "%d back-to-back replays, the last replay of each run read, medians"
                               % (ph["samples"], ph["replays_per_sample"]),
                        "step_ms_with_event_nodes": ph["step_with_event_nodes"]}
    else:
        ms_norm = statistics.mean(e[0].elapsed_time(e[1]) for e in evs)
        ms_clip = statistics.mean(e[1].elapsed_time(e[2]) for e in evs)
        ms_noise = statistics.mean(e[2].elapsed_time(e[3]) for e in evs)
        if fused and args.prefill or exchange is not None:
            gemm_ms_avg = ms_clip
        else:
            gemm_ms_avg = statistics.mean(e[4].elapsed_time(e[5]) for e in evs)

    # dominant kernel: the tensor-core G^T A GEMM of the clipped sums, timed live (see above)
    achieved_tf = counts["acc_flops"] / (gemm_ms_avg * 1e-3) / 1e12
    roofline = {"kernel": "%s (%s)" % (
                    gemm_kernel_name(ds, reserve),
                    "dp_clip_accumulate_noise_grouped, Gaussian noise drawn in the epilogue"
                    if fused and not args.prefill else
                    "dp_clip_accumulate_grouped, accumulating onto noise filled beside the norm phase"
                    if fused else "dp_clip_accumulate_grouped"),
                "bound": "tensor",
                "achieved": achieved_tf, "peak": peak_tf, "unit": "TFLOP/s",
                "frac": achieved_tf / peak_tf,
                "peak_source": "%s %s bf16 peak: %s" % (peaks["source"], peak_kind, peak_why),
                "frac_of_burst_peak": achieved_tf / peaks["bf16_tflops"],
                "frac_of_sustained_peak": achieved_tf / peaks["bf16_tflops_sustained"],
                # the burst peak scaled to the SM clock sampled during this timed region: what the
                # same tensor cores deliver at the clock the power cap left them
                "frac_of_burst_peak_at_sampled_clock": (
                    achieved_tf / (peaks["bf16_tflops"] * clocks["sm_mhz"] / clocks["sm_max_mhz"])
                    if clocks and clocks.get("sm_mhz") and clocks.get("sm_max_mhz") else None),
                "launches_per_step": 1 if exchange is None else 4, "ms_per_launch_avg": gemm_ms_avg,
                "timed_bracket": ("the grouped GEMM call" if exchange is None else
                                  "the whole clip phase (four GEMM launches, scatters, vectors): N > 1"),
                "flops_per_launch": counts["acc_flops"],
                "traffic": int(GEMM_DRAM_OVER_ALGORITHMIC * counts["acc_bytes"]),
                "traffic_how": ("%.2f x the launch's algorithmic bytes (%d): DRAM read + write of one ncu "
                                "capture of a three-wave, head-like launch of this kernel, scaled by bytes"
                                % (GEMM_DRAM_OVER_ALGORITHMIC, counts["acc_bytes"]))}
    ghost = ghost_norm_alone(dp, ds, peaks, peak_tf, counts)
    big = ds.outs["wte"]
    noise_n = big.numel()
    noise_fn = lambda: dp.dp_add_noise(big, ds.sigma, ds.C, 1.0, args.seed, 0, 0)   # noqa: E731
    noise_ms = time_graph(noise_fn, reps=5)
    # the pass is bound by instruction issue, so it follows the SM clock: right after the timed
    # steps the clock is what the power cap left of it; after a pause it is the idle boost clock
    time.sleep(1.5)
    noise_ms_rested = time_graph(noise_fn, reps=20)
    others = {
        "%s (dp_ghost_norms)" % ghost["kernel"]: ghost,
        "add_noise_kernel (dp_add_noise, %d elements)" % noise_n: {
            "bound": "hbm", "note": "bound by instruction issue in practice (about 39 per element)",
            "ms": noise_ms,
            "achieved_GBs": 8 * noise_n / (noise_ms * 1e-3) / 1e9,
            "peak_GBs": peaks["hbm_gbs"], "frac": 8 * noise_n / (noise_ms * 1e-3) / 1e9 / peaks["hbm_gbs"],
            "ms_after_1p5s_pause": noise_ms_rested,
            "achieved_GBs_after_pause": 8 * noise_n / (noise_ms_rested * 1e-3) / 1e9,
            "frac_after_pause": 8 * noise_n / (noise_ms_rested * 1e-3) / 1e9 / peaks["hbm_gbs"]},
    }

    # end to end through the public API with HOST buffers: every step copies the step's inputs
    # from pinned host memory and reads the per-example norms and clip factors back
    lin_layers = ds.linears + ([ds.lm] if ds.lm else [])
    host_in, dev_in = [], []
    seen = set()
    e2e_enabled = ds.input_bytes() < 12e9 and not args.device_inputs
    for t in ([ds.ids, ds.G_emb] + [x for l in lin_layers for x in (l.A, l.G)]) if e2e_enabled else []:
        if t.data_ptr() in seen:
            continue
        seen.add(t.data_ptr())
        h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
        h.copy_(t)
        host_in.append(h); dev_in.append(t)
    host_out = torch.empty(2, w.B, dtype=torch.float32, pin_memory=True)
    h2d = sum(h.numel() * h.element_size() for h in host_in)
    d2h = host_out.numel() * 4

    def e2e_step(k):
        for h, t in zip(host_in, dev_in):
            t.copy_(h, non_blocking=True)
        step(k)
        host_out[0].copy_(ds.norms, non_blocking=True)
        host_out[1].copy_(ds.clip, non_blocking=True)
        torch.cuda.synchronize()

    e2e_val, e2e_steps = None, 0
    if e2e_enabled:
        e2e_steps = max(3, min(args.steps, 10))
        e2e_step(0)
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for k in range(e2e_steps):
            e2e_step(k)
        t_e2e = time.perf_counter() - t0
        if world > 1:
            t = torch.tensor([t_e2e], device=dev)
            dist.all_reduce(t, op=dist.ReduceOp.MAX)
            t_e2e = float(t.item())
        e2e_val = world * w.B * e2e_steps / t_e2e
    del host_in

    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return

    # CPU baseline: the oracle on a bounded sample, on this machine's host cores (rank 0, N=1 only)
    cpu = None
    if world == 1 and not args.no_cpu_baseline and not args.device_inputs:
        t1 = oracle_sample_step(w, 1)
        n_ex = max(1, min(w.B, 16, int(20.0 / max(t1, 1e-3))))       # about 20 s of oracle work
        t_ex = oracle_sample_step(w, n_ex)
        n_noise = 4_000_000
        t_noise = oracle_noise_seconds(n_noise)
        est_step = t_ex * (w.B / n_ex) + t_noise * (counts["n_params"] / n_noise)
        cpu = {"value": w.B / est_step, "unit": UNIT, "cores": len(os.sched_getaffinity(0)),
               "kind": "oracle",
               "sample": (f"{n_ex} of {w.B} examples through norms+clip+sums of all layers "
                          f"({t_ex:.1f} s) and noise on {n_noise} of {counts['n_params']} parameters "
                          f"({t_noise:.1f} s), scaled to one full step ({est_step:.1f} s)")}

    # the same step issued call by call (no graph), for comparison
    graph_info = None
    if use_graph:
        n_eager = min(args.steps, 100)
        for k in range(3):
            eager_step(k)
        q0, q1 = _ev(), _ev()
        torch.cuda.synchronize()
        q0.record(stream)
        for k in range(n_eager):
            eager_step(k)
        q1.record(stream)
        torch.cuda.synchronize()
        e_ms = q0.elapsed_time(q1) / n_eager
        assert int(ds.dev_status.item()) == 0, "device status flagged a problem in the eager steps"
        graph_info = {"timed_region": "replays of pipeline.StepGraph (one CUDA graph launch per step)",
                      "kernels_per_replay": int(sg.kernels_per_replay),
                      "eager_ms_per_step": e_ms, "eager_value": w.B / (e_ms * 1e-3), **graph_detail}
    memory = {"max_allocated_bytes": int(torch.cuda.max_memory_allocated(dev)),
              "input_bytes": int(ds.input_bytes())}

    # ghost vs direct per layer shape of this workload, the other configurations, the tied path
    modes = sweep = tied_cost = None
    if world == 1 and not args.no_sweep and w.dtype == "bf16":
        modes = norm_modes(dp, ds, peaks)
        # free this workload's tensors first: the largest sweep cell needs ~25 GB by itself
        n_lin, has_lm, n_vec = len(w.linears), bool(w.lm), len(getattr(w, "vectors", []) or [])
        sg = None
        eager_step = step = e2e_step = None
        del ds, lin_layers, dev_in, big
        torch.cuda.empty_cache()
        sweep, tied_cost = run_sweep(P, dp, peaks, sampler, args.seed)
    else:
        n_lin, has_lm, n_vec = len(w.linears), bool(w.lm), len(getattr(w, "vectors", []) or [])
    if sampler:
        sampler.stop()

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": w.dtype, "data": "synthetic",
        "config": {"workload": w.name, "B_per_gpu": w.B, "T": w.T, "V": w.V, "layers": n_lin,
                   "lm_head": has_lm, "tied": w.tied, "positions": w.positions,
                   "bias_and_layernorm_params": n_vec,
                   "accumulate": "fp32", "input_bytes_per_step": memory["input_bytes"],
                   "exchange": (args.exchange + (" + all_gather" if args.gather else "")) if world > 1 else None,
                   "reserved_sms": reserve,
                   "l2": "inputs (%.2f GB per step) are larger than the 126 MB L2" % (memory["input_bytes"] / 1e9)},
        "phases_ms": {"norms": ms_norm, "clip_accumulate": ms_clip, "noise": ms_noise,
                      "norm_plus_clip": ms_norm + ms_clip,
                      "noise_fused_into_clip_accumulate": fused},
        "gpu_launches": int(launches),
        "cuda_graph": graph_info if graph_info is not None else (
            {"timed_region": graph_note} if graph_note else None),
        "memory": memory,
        "clocks": clocks,
        "roofline": roofline,
        "roofline_other": others,
        "e2e": ({"value": e2e_val, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
                 "d2h_bytes_per_step": int(d2h), "steps": e2e_steps} if e2e_enabled else None),
        "cpu_baseline": cpu,
        "norm_modes": modes,
        "tied_extra_cost": tied_cost,
        "sweep": sweep,
        "exchange_bytes_per_rank_per_step": exchange.bytes_on_wire if exchange is not None else None,
        "peaks": peaks,
    }
    print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


# ------------------------------------------------- small single-entry-point cases (profilers)
def run_case(args):
    """One entry point a few times on a small case: inputs larger than the 126 MB L2 but well
    under a few GB, so that a multi-pass profiler capture stays short.  Prints one JSON line."""
    import torch

    from paper_2609_40335_b200 import binding as dp

    torch.cuda.set_device(0)
    torch.manual_seed(0)
    dp.load()
    reps = args.reps

    def rb(*shape, std=1.0):
        return (torch.randn(*shape, device="cuda") * std).to(torch.bfloat16)

    def timed(fn):
        # device time per call: `reps` calls captured in one CUDA graph (host work stays outside)
        return time_graph(fn, reps)

    out = {"case": args.case, "reps": reps}
    c = args.case
    if c in ("gemm", "gemm_unclipped", "gemm_noise", "gemm_head"):
        # three full waves of 256 x 256 output tiles on 74 CTA pairs.  gemm*: a block-like layer
        # 1536 -> 9472 at B=64, T=128 (clip factors applied inside the pipeline); gemm_head: a
        # head-like layer 768 -> 18944 at B=32 (its narrow operand is scaled in a pass of its own)
        B, T, d_, p_ = (32, 128, 768, 148 * 128) if c == "gemm_head" else (64, 128, 1536, 37 * 256)
        L = [dp.Linear(rb(B, T, d_), rb(B, T, p_, std=1e-2))]
        outs = [torch.empty(p_, d_, device="cuda")]
        sq = torch.full((B,), 1e-12 if c == "gemm_unclipped" else 4.0, device="cuda")
        if c == "gemm_noise":
            ms = timed(lambda: dp.dp_clip_accumulate_noise_grouped(L, B, T, sq, 1.0, outs, 0.8, 1.0, 0, [0], 0))
        else:
            ms = timed(lambda: dp.dp_clip_accumulate_grouped(L, B, T, sq, 1.0, outs))
        out.update(ms=ms, TFLOPs=2 * B * T * d_ * p_ / ms / 1e9)
    elif c == "direct":
        # DIRECT norm (gradient tiles in tensor memory, square-sum epilogue): 768 -> 3072, T = 256
        B, T = 64, 256
        L = [dp.Linear(rb(B, T, 768), rb(B, T, 3072, std=1e-2), mode=dp.DP_NORM_DIRECT) for _ in range(4)]
        sq = torch.zeros(B, device="cuda")
        ms = timed(lambda: dp.dp_ghost_norms(L, B, T, sq))
        out.update(ms=ms, TFLOPs=len(L) * 2 * B * T * 768 * 3072 / ms / 1e9)
    elif c == "ghost":
        B, T = 32, 128
        L = [dp.Linear(rb(B, T, 768), rb(B, T, 3072, std=1e-2)) for _ in range(6)]
        L.append(dp.Linear(rb(B, T, 768), rb(B, T, 16384, std=1e-2)))
        sq = torch.zeros(B, device="cuda")
        ms = timed(lambda: dp.dp_ghost_norms(L, B, T, sq))
        out.update(ms=ms, GBs=sum(2 * B * T * (l.A.shape[-1] + l.G.shape[-1]) for l in L) / ms / 1e6)
    elif c == "ghost512":
        B, T = 64, 512
        L = [dp.Linear(rb(B, T, 1024), rb(B, T, 4096, std=1e-2)) for _ in range(2)]
        sq = torch.zeros(B, device="cuda")
        ms = timed(lambda: dp.dp_ghost_norms(L, B, T, sq))
        out.update(ms=ms, TFLOPs_needed=len(L) * B * T * (T + 1) * 5120 / ms / 1e9,
                   GBs=len(L) * B * 2 * T * 5120 / ms / 1e6)
    elif c == "ghost256":
        # T = 256: one diagonal 256 x 256 tile pair per (example, layer), the HBM-bound regime of
        # the CTA-pair kernel
        B, T = 64, 256
        L = [dp.Linear(rb(B, T, 768), rb(B, T, 3072, std=1e-2)) for _ in range(6)]
        sq = torch.zeros(B, device="cuda")
        ms = timed(lambda: dp.dp_ghost_norms(L, B, T, sq))
        out.update(ms=ms, GBs=len(L) * B * 2 * T * 3840 / ms / 1e6,
                   TFLOPs_needed=len(L) * B * T * (T + 1) * 3840 / ms / 1e9)
    elif c == "noise":
        x = torch.zeros(50257 * 768, device="cuda")
        ms = timed(lambda: dp.dp_add_noise(x, 0.8, 1.0, 1.0, 1234, 0, 0))
        out.update(ms=ms, GBs=8 * x.numel() / ms / 1e6)
    elif c in ("embed", "embed_small"):
        B, T, d, V = (256, 512, 1024, 50257) if c == "embed" else (32, 128, 768, 50257)
        w = torch.arange(1, V + 1, device="cuda", dtype=torch.float64) ** -1.1
        ids = torch.multinomial(w / w.sum(), B * T, replacement=True).to(torch.int32).view(B, T)
        G = rb(B, T, d, std=1e-2)
        sq = torch.zeros(B, device="cuda")
        o = torch.empty(V, d, device="cuda")

        def both():
            dp.dp_embed_norms(ids, G, V, sq)
            dp.dp_clip_accumulate_embed(ids, G, V, sq, 1.0, o)
        out.update(ms=timed(both))
    elif c == "cross":
        B, T, d, V = 32, 128, 768, 50257
        ids = torch.randint(0, V, (B, T), device="cuda", dtype=torch.int32)
        Ge, Al, Gl = rb(B, T, d, std=1e-2), rb(B, T, d), rb(B, T, 50264, std=1e-2)
        sq = torch.zeros(B, device="cuda")
        out.update(ms=timed(lambda: dp.dp_tied_cross_term(ids, Ge, Al, Gl, V, sq=sq, d=d)))
    elif c == "vectors":
        B, T = 32, 128
        vec = []
        for _ in range(6):
            for p_, with_x in [(768, True), (768, False), (2304, False), (768, False), (768, True),
                               (768, False), (3072, False), (768, False)]:
                vec.append(dp.Vector(rb(B, T, p_, std=1e-2), rb(B, T, p_) if with_x else None, p=p_))
        sq = torch.zeros(B, device="cuda")
        outs = [torch.empty(v.p, device="cuda") for v in vec]

        def both():
            dp.dp_vector_norms(vec, B, T, sq)
            dp.dp_clip_accumulate_vectors(vec, B, T, sq, 1.0, outs)
        out.update(ms=timed(both))
    elif c == "f32":
        # fp32 inputs: the two-term bf16 split on the tensor cores against the plain fp32-FMA kernels
        # (norm in both modes, clipped sum), 768 -> 3072 at B = 8, T = 128
        B, T, d_, p_ = 8, 128, 768, 3072
        A, G = torch.randn(B, T, d_, device="cuda"), torch.randn(B, T, p_, device="cuda") * 1e-2
        sq = torch.zeros(B, device="cuda")
        o = torch.empty(p_, d_, device="cuda")
        clipsq = torch.full((B,), 4.0, device="cuda")
        for name, on in (("tensor", False), ("fma", True)):
            dp.dp_debug_force_fma(on)
            for mode, key in ((dp.DP_NORM_GHOST, "ghost"), (dp.DP_NORM_DIRECT, "direct")):
                L = [dp.Linear(A, G, mode=mode)]
                out[f"{name}_{key}_norm_ms"] = timed(lambda: dp.dp_ghost_norms(L, B, T, sq))
            out[f"{name}_clipped_sum_ms"] = timed(lambda: dp.dp_clip_accumulate(A, G, clipsq, 1.0, o))
        dp.dp_debug_force_fma(False)
        out["clipped_sum_TFLOPs_fp32_equivalent"] = 2 * B * T * d_ * p_ / out["tensor_clipped_sum_ms"] / 1e9
    else:
        raise SystemExit("unknown --case %r" % c)
    print(json.dumps(out), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    # default: enough back-to-back steps (about two seconds) for the SM clock to settle under the
    # power cap; the reference arm, whose steps take seconds each, defaults to 20
    ap.add_argument("--steps", type=int, default=None)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--exchange", default="reduce_scatter", choices=["all_reduce", "reduce_scatter"],
                    help="N > 1: bucketed reduce-scatter on a communication stream, noise on the owned "
                         "slice (default), or a blocking all-reduce per tensor followed by the noise pass")
    ap.add_argument("--gather", action="store_true",
                    help="N > 1, reduce_scatter: all-gather the noised slices back into the full tensors")
    ap.add_argument("--reserve-sms", type=int, default=None,
                    help="SMs left free of the library's persistent kernels (default: 0 at N = 1, "
                         "NCCL_MAX_CTAS = 16 at N > 1, for the collectives)")
    ap.add_argument("--bucketed", action="store_true",
                    help="N = 1: run the multi-GPU step order (clipped sums bucket by bucket through the "
                         "exchange object, noise on the communication stream) on one GPU")
    ap.add_argument("--eager", action="store_true",
                    help="issue the step call by call instead of replaying a captured CUDA graph")
    ap.add_argument("--workload", default="cfg3")
    ap.add_argument("--B", type=int, default=0, help="override the workload's batch size (cfg5 sweep)")
    ap.add_argument("--T", type=int, default=0, help="override the workload's sequence length")
    ap.add_argument("--full-model", action="store_true",
                    help="also clip the biases and LayerNorm parameters of every block (whole GPT-2 model)")
    ap.add_argument("--device-inputs", action="store_true",
                    help="cfg5 only: draw the inputs on the device (big cells)")
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-sweep", action="store_true",
                    help="skip the sweep over the other configurations, norm_modes and the tied cost")
    ap.add_argument("--prefill", action="store_true", help="noise of every tensor filled beside the norms")
    ap.add_argument("--unfused", action="store_true",
                    help="separate noise pass instead of fused noise (N = 1)")
    ap.add_argument("--case", default=None, help="run one small single-entry-point case and exit")
    ap.add_argument("--reps", type=int, default=3)
    args = ap.parse_args()
    if args.case:
        run_case(args)
        return
    if args.steps is None:
        args.steps = 20 if args.impl == "reference" else 400
    if args.impl == "reference":
        run_reference(args)      # any K: the per-step sample shrinks so that the run stays bounded
    else:
        if args.warmup < 3:
            args.warmup = 3
        run_ours(args)


if __name__ == "__main__":
    main()
