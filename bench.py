#!/usr/bin/env python
"""Benchmark: full-size six-hour latent rollout step of the WeatherMesh-3 processor.

Workload (one "step" = one forecast): one six-hour processor call (8 blocks)
on a 9 x 90 x 180 latent (145,800 tokens) with C = 768, 16 heads and a
5 x 7 x 7 neighborhood window, BF16 tensor-core path with FP32 accumulation
and FP32 residual stream; seeded synthetic latent ~ N(0,1) and Xavier-uniform
random weights (the paper's trained weights and ERA-5 data are not available).
Metric: forecasts/s (six-hour latent forecasts of the full-size latent).

Also measured: the plain FP32 GPU path on the same step and its BF16-vs-FP32
error, an end-to-end number through the host-buffer C-ABI call, the dominant
kernel's roofline fraction from per-launch CUDA events, the 14-day rollout on
the 4 x 24 x 48 x 128 latent, serving, and the FP64 CPU oracle timed on a
bounded sample. One JSON line on stdout holds the result and the main figure of
each of these; the whole record, with every list, is a JSON line on stderr.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
Multi-GPU (replicas, weak scaling): torchrun --nproc-per-node N bench.py --gpus N ...
"""
from __future__ import annotations

import argparse
import dataclasses
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import synth  # noqa: E402

METRIC = "latent-rollout forecasts/s (full-size six-hour step)"
UNIT = "forecasts/s"
WORKLOAD = "six-hour processor step, 8 blocks, latent 9x90x180x768 (145,800 tokens), 16 heads, window 5x7x7"
# bounded CPU-oracle sample: a latitude band of the same latent (all levels,
# 7 latitudes, 80 longitudes); every token has the same per-token work
# (full 5x7x7 bump window, C = 768) as in the full latent
CPU_SAMPLE = dataclasses.replace(synth.FULL, H=7, W=80)


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return {"hbm_gbs": d.get("hbm_gbs", 6800.0), "bf16_tflops": d.get("bf16_tflops", 1900.0),
                "bf16_tflops_sustained": d.get("bf16_tflops_sustained", 1700.0), "source": "measured"}
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "source": "fallback"}


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *a):
        self.lines = []
        if self.proc is not None:
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                out, _ = self.proc.communicate()
            self.lines = [ln for ln in out.splitlines() if ln.strip()]

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in getattr(self, "lines", []):
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def _capture(kind, field="dram_bytes_per_launch"):
    """A per-launch counter of this kernel from the committed ncu summary
    (DRAM bytes, warp instructions), or None when the kernel source has
    changed since that capture."""
    import hashlib
    p = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p):
        return None
    with open(p) as f:
        d = json.load(f).get(kind)
    if not d or field not in d:
        return None
    with open(os.path.join(ROOT, d["source"]), "rb") as f:
        if hashlib.sha256(f.read()).hexdigest() != d["source_sha256"]:
            return None
    return d[field]


def _traffic(kind):
    return _capture(kind, "dram_bytes_per_launch")


def max_over_ranks(x: float, device) -> float:
    """Largest x over the ranks of the default process group (x itself when single)."""
    import torch
    import torch.distributed as dist
    if not dist.is_available() or not dist.is_initialized() or dist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_value(local_total_ms: float, steps: int, world_size: int, device) -> tuple[float, float]:
    """(slowest rank's total ms, whole-job forecasts/s) for `steps` steps on every replica."""
    total_ms = max_over_ranks(local_total_ms, device)
    return total_ms, world_size * steps / (total_ms / 1e3)


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def _small_block_seconds(threads=None) -> float:
    """Seconds per FP64 oracle block on the small latent (4x24x48x128), timed in
    a fresh interpreter whose BLAS runs `threads` threads (None: its default)."""
    code = ("import sys, time; sys.path.insert(0, %r); import synth; from oracle import wm_oracle as orc; "
            "s = synth.SMALL; x = synth.latent(s, 1, 1); w = synth.block_weights(s.C, 0, 0, 0); orc.block(x, w, s); "
            "t = time.perf_counter(); [orc.block(x, w, s) for _ in range(3)]; "
            "print((time.perf_counter() - t) / 3)") % ROOT
    env = dict(os.environ)
    if threads:
        for var in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
            env[var] = str(threads)
    out = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=600)
    return float(out.stdout.strip().splitlines()[-1])


def cpu_oracle_baseline(seconds_budget: float = 12.0, sample=CPU_SAMPLE):
    """Time the FP64 oracle on a bounded band of the workload; scale to forecasts/s."""
    from oracle import wm_oracle as orc
    x = synth.latent(sample, 1, seed=1)
    w = synth.block_weights(sample.C, 0, 0, 0)
    t0 = time.perf_counter()
    reps = 0
    while True:
        orc.block(x, w, sample)
        reps += 1
        if time.perf_counter() - t0 > seconds_budget or reps >= 8:
            break
    dt = (time.perf_counter() - t0) / reps
    per_token = dt / sample.N
    sec_per_forecast = per_token * synth.FULL.N * synth.FULL.blocks_p6
    return {"value": 1.0 / sec_per_forecast, "unit": UNIT, "cores": os.cpu_count(), "kind": "oracle",
            "sample": (f"one block on a {sample.D}x{sample.H}x{sample.W}x{sample.C} latitude band of the latent "
                       f"({sample.N} tokens, x{reps}), {dt:.2f} s per block, scaled by tokens to 8 blocks x "
                       f"{synth.FULL.N} tokens; numpy float64, BLAS multi-threaded, gathers single-threaded"),
            "seconds_per_forecast": sec_per_forecast,
            "small_latent": _small_latent_cpu()}


def _small_latent_cpu():
    """The small latent's oracle block on one thread and on every core, and
    the 14-day rollout (448 blocks) those times imply."""
    try:
        one, allc = _small_block_seconds(1), _small_block_seconds(None)
    except (subprocess.SubprocessError, ValueError, IndexError) as e:
        return {"error": str(e)[:200]}
    return {"workload": "one block, latent 4x24x48x128, window 3x5x5", "block_s_1_thread": one,
            "block_s_all_cores": allc, "cores": os.cpu_count(),
            "rollout_336h_s_1_thread": 448 * one, "rollout_336h_s_all_cores": 448 * allc}


ORACLE_ROLLOUT_THREADS = 8


def start_oracle_rollout(lead=337):
    """CPU-baseline leg: the FP64 oracle's 14-day rollout of the small latent
    (4x24x48x128; 56 six-hour + 1 one-hour steps, 452 blocks), timed in a
    fresh interpreter on ORACLE_ROLLOUT_THREADS host threads while the GPU
    sections run. Its per-step latents are the reference of the rollout error
    curve. Returns the running process and the file it writes."""
    import tempfile
    fd, path = tempfile.mkstemp(suffix=".npz", prefix="wm_oracle_rollout_")
    os.close(fd)
    code = ("import sys, time; sys.path.insert(0, %r); import numpy as np; import synth; "
            "from oracle import wm_oracle as orc; s = synth.SMALL; p6, p1 = synth.processor_weights(s, seed=0); "
            "x = synth.latent(s, 1, seed=1); steps = []; t = time.perf_counter(); "
            "orc.rollout(x, %d, p6, p1, s, per_step=steps); dt = time.perf_counter() - t; "
            "np.savez(%r, steps=np.stack(steps), seconds=dt)") % (ROOT, lead, path)
    env = dict(os.environ)
    for var in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        env[var] = str(ORACLE_ROLLOUT_THREADS)
    proc = subprocess.Popen([sys.executable, "-c", code], env=env, stdout=subprocess.DEVNULL,
                            stderr=subprocess.PIPE, text=True)
    return proc, path


def finish_oracle_rollout(proc, path, timeout=900):
    """(per-step oracle latents [steps, 1, D, H, W, C] float64, seconds) or (None, error text)."""
    try:
        _, err = proc.communicate(timeout=timeout)
        if proc.returncode != 0:
            return None, (err or "")[-300:]
        with np.load(path) as z:
            return z["steps"], float(z["seconds"])
    except subprocess.TimeoutExpired:
        proc.kill()
        return None, "timed out"
    finally:
        if os.path.exists(path):
            os.remove(path)


def rollout_error_curve(wm, torch, dev, oracle_steps, lead=337):
    """Relative L2 error against the FP64 oracle after every processor step of
    the 337-hour rollout (small latent; the 336-hour forecast is step 56) in
    FP32, BF16 and FP8-MLP. Each step runs through wm_processor_step on the
    device; the comparison is in float64 on the host."""
    s = synth.SMALL
    p6, p1 = synth.processor_weights(s, seed=0)
    n6, n1 = divmod(lead, 6)
    ctx = wm.wm_create_from_host(wm.make_config(s, wm.WM_PREC_BF16), synth.pack_weights(p6, p1))
    res = {"workload": f"latent 4x24x48x128, {lead} h = {n6} six-hour + {n1} one-hour steps "
                       f"({n6 * s.blocks_p6 + n1 * s.blocks_p1} blocks), relative L2 vs the FP64 oracle after each step"}
    try:
        for prec, name in ((wm.WM_PREC_FP32, "fp32"), (wm.WM_PREC_BF16, "bf16"), (wm.WM_PREC_BF16_FP8MLP, "fp8mlp")):
            wm.wm_set_precision(ctx, prec)
            x = torch.from_numpy(synth.latent(s, 1, seed=1)).to(dev)
            errs = []
            for k in range(n6 + n1):
                wm.wm_processor_step(ctx, x, wm.WM_P6 if k < n6 else wm.WM_P1)
                got = x.detach().cpu().numpy().astype(np.float64)
                ref = oracle_steps[k]
                errs.append(float(np.linalg.norm(got - ref) / np.linalg.norm(ref)))
            res[name] = {"per_step": errs, "after_step_1": errs[0], "final_336h": errs[n6 - 1],
                         "final_337h": errs[-1], "max": max(errs),
                         "nonfinite_final": wm.wm_count_nonfinite(x)}
    finally:
        wm.wm_destroy(ctx)
    return res


def run_reference(args):
    """The reference arm: the FP64 CPU oracle on the host cores. Each step is
    one processor block on a 9 x 7 x 20 latitude band of the full-size latent
    (1,260 tokens; every token has the full 5 x 7 x 7 window and C = 768, so
    the per-token work is the full latent's). ms_per_step is that band's
    measured time; value scales it by tokens and blocks to full-size six-hour
    forecasts/s, the unit of the GPU line."""
    ws, rank, _ = _dist()
    if rank != 0:
        return
    sample = dataclasses.replace(synth.FULL, H=7, W=20)
    from oracle import wm_oracle as orc
    x = synth.latent(sample, 1, seed=1)
    w = synth.block_weights(sample.C, 0, 0, 0)
    for _ in range(args.warmup):
        orc.block(x, w, sample)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        orc.block(x, w, sample)
    dt = (time.perf_counter() - t0) / args.steps
    sec_per_forecast = dt / sample.N * synth.FULL.N * synth.FULL.blocks_p6
    value = 1.0 / sec_per_forecast
    band = (f"one block on a {sample.D}x{sample.H}x{sample.W}x{sample.C} latitude band ({sample.N} tokens) of the "
            f"9x90x180x768 latent")
    desc = f"per step {band}; value scaled by tokens ({synth.FULL.N}) and blocks ({synth.FULL.blocks_p6})"
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 0, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": dt * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": f"FP64 oracle, {band}, scaled to the {WORKLOAD}",
                       "timed_per_step": band, "ms_per_full_forecast": sec_per_forecast * 1e3,
                       "impl_note": "FP64 CPU oracle (numpy) on host cores"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": os.cpu_count(), "kind": "oracle",
                             "sample": desc},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_ours(args):
    import torch
    import paper_2503_22235_gb300 as wm
    from paper_2503_22235_gb300 import build as wm_build

    ws, rank, local = _dist()
    oracle_job = start_oracle_rollout() if (rank == 0 and ws == 1 and not args.no_cpu) else None
    torch.cuda.set_device(local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    wm_build.build()
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream()

    shape = synth.FULL
    p6, p1 = synth.processor_weights(shape, seed=0)
    ctx = wm.wm_create_from_host(wm.make_config(shape, wm.WM_PREC_BF16), synth.pack_weights(p6, p1))
    x0 = synth.latent(shape, 1, seed=1 + rank)
    x = torch.from_numpy(x0).to(dev)

    def barrier():
        if ws > 1:
            torch.distributed.barrier()

    # ---------------- warm-up
    for _ in range(args.warmup):
        wm.wm_processor_step(ctx, x, wm.WM_P6)
    torch.cuda.synchronize()

    # ---------------- timed region: K six-hour steps, per-launch events for the roofline
    wm.wm_timing_begin(ctx, max_launches=7 * shape.blocks_p6 * args.steps + 16)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clk:
        barrier()
        torch.cuda.synchronize()
        ev0.record(stream)
        for _ in range(args.steps):
            wm.wm_processor_step(ctx, x, wm.WM_P6)
        ev1.record(stream)
        torch.cuda.synchronize()
        barrier()
    kt = wm.wm_timing_end(ctx)
    wm.wm_device_status()
    total_ms, value = replica_value(ev0.elapsed_time(ev1), args.steps, ws, dev)
    ms_per_step = total_ms / args.steps
    launches = sum(c for _, c in kt.values())

    # ---------------- roofline of the dominant kernel (and of every GEMM)
    peaks = _peaks()
    M, C = shape.N, shape.C
    K = shape.kd * shape.kh * shape.kw
    flops = {"qkv": 2.0 * M * C * 3 * C, "proj": 2.0 * M * C * C, "fc1": 2.0 * M * C * 4 * C,
             "fc2": 2.0 * M * 4 * C * C, "attn": 4.0 * M * K * C}
    # algorithmic HBM bytes: attention reads q, k, v and writes o (bf16, 8C per
    # token); LayerNorm reads the fp32 row and writes the bf16 row (6C)
    hbm_bytes = {"attn": 8.0 * M * C, "ln1": 6.0 * M * C, "ln2": 6.0 * M * C}
    dom = max((k for k in kt if kt[k][1] > 0), key=lambda k: kt[k][0])
    avg_ms = kt[dom][0] / kt[dom][1]
    traffic = _traffic(dom)
    if dom in hbm_bytes and flops.get(dom, 0.0) / hbm_bytes[dom] < peaks["bf16_tflops"] * 1e3 / peaks["hbm_gbs"]:
        achieved = hbm_bytes[dom] / (avg_ms * 1e-3) / 1e9
        roofline = {"bound": "hbm", "kernel": dom, "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                    "frac": achieved / peaks["hbm_gbs"], "traffic": traffic,
                    "algorithmic_bytes_per_launch": hbm_bytes[dom],
                    "peak_source": f"{peaks['source']} HBM copy bandwidth"}
    else:
        achieved = flops[dom] / (avg_ms * 1e-3) / 1e12
        roofline = {"bound": "tensor", "kernel": dom, "achieved": achieved, "peak": peaks["bf16_tflops_sustained"],
                    "unit": "TFLOP/s", "frac": achieved / peaks["bf16_tflops_sustained"], "traffic": traffic,
                    "peak_source": f"{peaks['source']} bf16 sustained (kernel timed inside a long step)"}
    roofline["avg_launch_ms"] = avg_ms
    # Instruction-issue view: the attention kernel's limit is issuing its
    # softmax instructions, not DRAM. Warp instructions per launch from the
    # ncu capture over the live launch time, against 4 schedulers x SMs x
    # the SM clock sampled during the timed region (one warp instruction per
    # scheduler per cycle).
    instr = _capture(dom, "warp_instructions_per_launch")
    clk_mhz = (clk.summary() or {}).get("sm_mhz") or 2070.0
    if instr:
        n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
        issue_peak = 4 * n_sm * clk_mhz * 1e6
        roofline["issue"] = {"warp_instructions_per_launch": instr,
                             "achieved_per_s": instr / (avg_ms * 1e-3), "peak_per_s": issue_peak,
                             "frac": instr / (avg_ms * 1e-3) / issue_peak,
                             "peak_source": f"4 warp schedulers x {n_sm} SMs x median SM clock under load"}
    roofline["kernels_ms_per_step"] = {k: v[0] / args.steps for k, v in kt.items()}
    roofline["gemm_tflops"] = {k: flops[k] / (kt[k][0] / kt[k][1] * 1e-3) / 1e12 for k in ("qkv", "proj", "fc1", "fc2")
                               if kt[k][1]}
    roofline["gemm_frac_of_sustained"] = {k: v / peaks["bf16_tflops_sustained"]
                                          for k, v in roofline["gemm_tflops"].items()}
    if kt["attn"][1]:
        roofline["attn_algorithmic_tflops"] = flops["attn"] / (kt["attn"][0] / kt["attn"][1] * 1e-3) / 1e12

    out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
           "config": {"workload": WORKLOAD, "batch_per_gpu": 1, "blocks": shape.blocks_p6,
                      "parallelism": f"replicas x{ws}" if ws > 1 else "single GPU",
                      "l2": "working set larger than L2 (latent 448 MB fp32, activations ~2 GB bf16)"},
           "gpu_launches": launches, "clocks": clk.summary(), "roofline": roofline}

    # ---------------- FP32 plain path on the same step + BF16-vs-FP32 error
    if not args.no_fp32:
        xa = torch.from_numpy(x0).to(dev)
        xb = torch.from_numpy(x0).to(dev)
        wm.wm_processor_step(ctx, xa, wm.WM_P6)          # BF16
        wm.wm_set_precision(ctx, wm.WM_PREC_FP32)
        wm.wm_processor_step(ctx, xb, wm.WM_P6)          # FP32 (also warm-up)
        torch.cuda.synchronize()
        err = wm.wm_rel_l2(xa, xb)
        xc = torch.from_numpy(x0).to(dev)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        wm.wm_processor_step(ctx, xc, wm.WM_P6)
        e1.record(stream)
        torch.cuda.synchronize()
        fp32_ms = e0.elapsed_time(e1)
        # per-kernel times of one more FP32 step (CUDA events per launch)
        wm.wm_timing_begin(ctx, 8 * shape.blocks_p6 + 16)
        wm.wm_processor_step(ctx, xc, wm.WM_P6)
        torch.cuda.synchronize()
        f32_kt = wm.wm_timing_end(ctx)
        wm.wm_set_precision(ctx, wm.WM_PREC_BF16)
        # FP32 FMA peak (nominal): 128 FP32 lanes per SM, one FMA (2 flop) per lane per clock;
        # linear layers run as six bf16 tensor-core products each, against a sixth of the measured BF16 rate
        n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
        f32_peak = 2.0 * 128 * n_sm * ((clk.summary() or {}).get("sm_mhz") or 2070.0) * 1e6 / 1e12
        f32_tf = {k: flops[k] / (f32_kt[k][0] / f32_kt[k][1] * 1e-3) / 1e12
                  for k in ("qkv", "proj", "fc1", "fc2", "attn") if f32_kt[k][1]}
        f32_peaks = {k: f32_peak if k == "attn" else peaks["bf16_tflops_sustained"] / 6 for k in f32_tf}
        f32_dom = max((k for k in f32_kt if f32_kt[k][1] > 0), key=lambda k: f32_kt[k][0])
        out["fp32_plain"] = {"value": 1e3 / fp32_ms, "unit": UNIT, "ms_per_step": fp32_ms,
                             "bf16_vs_fp32_rel_l2": err, "speedup_bf16": fp32_ms / ms_per_step,
                             "kernels_ms_per_step": {k: v[0] for k, v in f32_kt.items() if v[1]},
                             "roofline": {"bound": "alu" if f32_dom == "attn" else "tensor", "kernel": f32_dom,
                                          "achieved": f32_tf.get(f32_dom),
                                          "peak": f32_peaks.get(f32_dom, f32_peak), "unit": "TFLOP/s",
                                          "frac": (f32_tf.get(f32_dom) or 0.0) / f32_peaks.get(f32_dom, f32_peak),
                                          "tflops": f32_tf,
                                          "frac_by_kernel": {k: v / f32_peaks[k] for k, v in f32_tf.items()},
                                          "peak_source": "attention: nominal FP32 FMA rate, 128 lanes x 2 flop x SMs "
                                                         "x median SM clock under load; linear layers (six bf16 "
                                                         "products for one FP32): a sixth of the measured sustained "
                                                         "BF16 rate (no TF32)"}}
        del xa, xb, xc

    # ---------------- FP8-MLP precision on the same step
    if not args.no_fp32:
        xa = torch.from_numpy(x0).to(dev)
        xb = torch.from_numpy(x0).to(dev)
        wm.wm_set_precision(ctx, wm.WM_PREC_BF16_FP8MLP)
        wm.wm_processor_step(ctx, xa, wm.WM_P6)              # warm-up (tunes nothing new)
        xa.copy_(torch.from_numpy(x0).to(dev))
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        wm.wm_processor_step(ctx, xa, wm.WM_P6)
        e1.record(stream)
        torch.cuda.synchronize()
        f8_ms = e0.elapsed_time(e1)
        # per-kernel times of one more FP8-MLP step on a copy (eager, CUDA events per launch)
        xt = xa.clone()
        wm.wm_timing_begin(ctx, 8 * shape.blocks_p6 + 16)
        wm.wm_processor_step(ctx, xt, wm.WM_P6)
        torch.cuda.synchronize()
        f8_kt = wm.wm_timing_end(ctx)
        del xt
        wm.wm_set_precision(ctx, wm.WM_PREC_FP32)
        wm.wm_processor_step(ctx, xb, wm.WM_P6)
        wm.wm_set_precision(ctx, wm.WM_PREC_BF16)
        torch.cuda.synchronize()
        out["fp8mlp"] = {"value": 1e3 / f8_ms, "unit": UNIT, "ms_per_step": f8_ms,
                         "fp8mlp_vs_fp32_rel_l2": wm.wm_rel_l2(xa, xb),
                         "kernels_ms_per_step": {k: v[0] for k, v in f8_kt.items() if v[1]},
                         "e4m3_tflops": {k: flops[k] / (f8_kt[k][0] / f8_kt[k][1] * 1e-3) / 1e12
                                         for k in ("fc1", "fc2") if f8_kt[k][1]}}
        del xa, xb

    # ---------------- end to end through the host-buffer C-ABI call
    if not args.no_e2e:
        # a stream of K forecasts from pinned host memory; each step uploads its
        # input and downloads its result inside the timed region
        hin = torch.from_numpy(x0).pin_memory()
        houts = [torch.empty_like(hin).pin_memory() for _ in range(2)]
        wm.wm_forecast_host_many(ctx, [hin] * max(3, args.warmup), [houts[i % 2] for i in range(max(3, args.warmup))], 6)
        with ClockSampler(local) as eclk:
            barrier()
            t0 = time.perf_counter()
            wm.wm_forecast_host_many(ctx, [hin] * args.steps, [houts[i % 2] for i in range(args.steps)], 6)
            dt = max_over_ranks(time.perf_counter() - t0, dev)
        for _ in range(max(1, args.warmup)):
            wm.wm_forecast_host(ctx, hin, houts[0], 6)
        barrier()
        t1 = time.perf_counter()
        for _ in range(args.steps):
            wm.wm_forecast_host(ctx, hin, houts[0], 6)
        dt1 = max_over_ranks(time.perf_counter() - t1, dev)
        nbytes = hin.numel() * 4
        out["e2e"] = {"value": ws * args.steps / dt, "unit": UNIT, "h2d_bytes_per_step": nbytes,
                      "d2h_bytes_per_step": nbytes, "call": "wm_forecast_host_many(lead 6 h, K forecasts)",
                      "clocks": eclk.summary(),
                      "single_call": {"value": ws * args.steps / dt1, "call": "wm_forecast_host(lead 6 h) x K"}}
    # ---------------- 0.25-degree fields -> 14-day forecast -> fields (encoder, rollout, decoder)
    if not args.no_fields and rank == 0:
        out["fields_14d_full"] = fields_bench(wm, torch, dev, ctx, shape)
    out["autotune"] = wm.wm_autotune_report().strip().splitlines()
    out["roofline"]["attn_halo"] = attn_halo(out["autotune"], shape)
    wm.wm_destroy(ctx)

    # ---------------- 14-day rollout on the small latent (whole rollout as one CUDA graph)
    if not args.no_rollout:
        out["rollout_14d_small"] = small_rollout(wm, torch, dev)

    if not args.no_batch:
        out["batch_uneven_small"] = batch_bench(wm, torch, dev)
        out.update(hourly_ensemble_bench(wm, torch, dev))

    if not args.no_serve and rank == 0:
        out["serve"] = serve_bench(wm, torch, n_requests=args.serve_requests, bf16_only=args.serve_bf16_only)

    if rank == 0 and ws == 1 and not args.no_cpu:
        out["cpu_baseline"] = cpu_oracle_baseline()
        steps, info = finish_oracle_rollout(*oracle_job)
        if steps is None:
            out["cpu_baseline"]["rollout_337h_small"] = {"error": info}
        else:
            out["cpu_baseline"]["rollout_337h_small"] = {
                "workload": "FP64 oracle rollout, latent 4x24x48x128, 337 h (452 blocks)", "seconds": info,
                "forecasts_per_s": 1.0 / info, "threads": ORACLE_ROLLOUT_THREADS}
            out["rollout_error_vs_oracle"] = rollout_error_curve(wm, torch, dev, steps)
    if rank == 0:
        print(json.dumps(out), file=sys.stderr, flush=True)   # the whole record
        print(json.dumps(result_line(out)), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()


# One figure of each further section for the result line; the sections are in the record.
SECTION_FIGURES = {
    "fp32_plain": ("value", "bf16_vs_fp32_rel_l2"),
    "fp8mlp": ("value", "fp8mlp_vs_fp32_rel_l2"),
    "fields_14d_full": ("encode_ms", "decode_ms", "forecasts_per_s"),
    "rollout_14d_small": ("bf16_T336_forecasts_per_s", "bf16_batch4_T336_forecasts_per_s"),
    "batch_uneven_small": ("bf16_forecasts_per_s",),
    "hourly_small_14d": ("forecast_sets_per_s",),
    "ensemble_small_14d": ("member_forecasts_per_s",),
    "ensemble_full_6h": ("member_forecasts_per_s",),
    "serve": ("bf16_p50_ms", "bf16_p99_ms", "bf16_saturated_forecasts_per_s"),
}


def result_line(out):
    """The one line on stdout: every key that says what was measured and how, and one or two figures of the further
    sections. Lists by step and by plan make the whole record some 25 KB, more than readers of a log's tail keep."""
    keys = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks")
    line = {k: out[k] for k in keys if k in out}
    if "e2e" in out:
        line["e2e"] = {k: v for k, v in out["e2e"].items() if k not in ("clocks", "single_call")}
    line["roofline"] = {k: v for k, v in out["roofline"].items()
                        if k in ("bound", "kernel", "achieved", "peak", "unit", "frac", "traffic", "peak_source",
                                 "kernels_ms_per_step")}
    for name, figures in SECTION_FIGURES.items():
        if name in out:
            line[name] = {k: out[name][k] for k in figures if k in out[name]}
    curve = out.get("rollout_error_vs_oracle")
    if curve:
        line["rollout_error_vs_oracle"] = {prec: {k: r[k] for k in ("final_336h", "final_337h", "max")}
                                           for prec, r in curve.items() if isinstance(r, dict)}
    cpu = out.get("cpu_baseline")
    if cpu:
        line["cpu_baseline"] = {k: cpu[k] for k in ("value", "unit", "cores", "kind") if k in cpu}
    return line


def attn_halo(report, shape):
    """Scored keys per query and key level against the window's keys, for the
    attention plan the tuner kept at this shape (its line in the report:
    "... window=KDxKHxKW ... -> <family> ... patch=PHxPW ..."). A warp scores
    the rectangle (PH + kh - 1) x pow2(PW + kw - 1) for its PH x PW queries
    (16 queries, or 8 in the transposed family)."""
    import re
    win = f"window={shape.kd}x{shape.kh}x{shape.kw}"
    for line in report:
        if line.startswith("attention") and f"C={shape.C} " in line and win in line:
            m = re.search(r"patch=(\d+)x(\d+)", line)
            if not m:
                return None
            ph, pw = int(m.group(1)), int(m.group(2))
            span = 8
            while span < pw + shape.kw - 1:
                span *= 2
            issued = (ph + shape.kh - 1) * span
            useful = shape.kh * shape.kw
            return {"plan": line.split("->")[1].strip(), "scored_keys_per_query_level": issued,
                    "window_keys_per_level": useful, "scored_over_useful": issued / useful}
    return None


def fields_bench(wm, torch, dev, ctx, shape, lead=336, reps=2):
    """Encoder + 14-day latent rollout + decoder on the 0.25-degree grid (BF16)."""
    cd = synth.FULL_CODEC
    w = synth.codec_weights(cd, shape.C, seed=0)
    codec = wm.wm_codec_create(wm.make_codec_config(cd, shape.C, wm.WM_PREC_BF16), synth.pack_codec_weights(w))
    g = torch.Generator(device=dev)
    g.manual_seed(1)
    atm = torch.randn(cd.levels, cd.H0, cd.W0, cd.v_atm, device=dev, generator=g)
    sfc = torch.randn(cd.H0, cd.W0, cd.v_sfc_in, device=dev, generator=g)
    cst = torch.randn(cd.H0, cd.W0, cd.n_const, device=dev, generator=g)
    lat = torch.empty(cd.D, cd.H, cd.W, shape.C, device=dev)
    a_out = torch.empty(cd.levels, cd.H0, cd.W0, cd.v_atm, device=dev)
    s_out = torch.empty(cd.H0, cd.W0, cd.v_sfc_out, device=dev)
    stream = torch.cuda.current_stream()

    def timed(fn, n):
        fn()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(n):
            fn()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / n

    enc_ms = timed(lambda: wm.wm_encode(codec, atm, sfc, cst, lat), 3)
    dec_ms = timed(lambda: wm.wm_decode(codec, lat, a_out, s_out), 3)
    fc_ms = timed(lambda: wm.wm_forecast_fields(ctx, codec, atm, sfc, cst, lead, lat, a_out, s_out), reps)
    wm.wm_codec_destroy(codec)
    return {"workload": f"0.25-degree grid {cd.H0}x{cd.W0}: {cd.v_atm} atmospheric variables x {cd.levels} levels, "
                        f"{cd.v_sfc_in} surface inputs + {cd.n_const} constants -> {cd.v_sfc_out} surface outputs; "
                        f"encoder/decoder width {cd.Ce}, {cd.blocks} NA blocks each; lead {lead} h "
                        f"({lead // 6} six-hour steps); random fields", "precision": "bf16",
            "encode_ms": enc_ms, "decode_ms": dec_ms, "forecast_s": fc_ms / 1e3,
            "forecasts_per_s": 1e3 / fc_ms}


def small_rollout(wm, torch, dev, reps=10):
    """The 14-day rollout of the small latent: BF16 through the whole-rollout
    kernel (one launch) at batch 1 and 4, the same with the per-kernel path
    (one launch per GEMM / attention, captured as a graph), and FP32."""
    s = synth.SMALL
    p6, p1 = synth.processor_weights(s, seed=0)
    ctx = wm.wm_create_from_host(wm.make_config(s, wm.WM_PREC_BF16, 4), synth.pack_weights(p6, p1))
    x1 = torch.from_numpy(synth.latent(s, 1, seed=1)).to(dev)
    x4 = torch.from_numpy(synth.latent(s, 4, seed=1)).to(dev)
    res = {"workload": "latent 4x24x48x128, window 3x5x5, P6 8 blocks + P1 4 blocks, greedy schedule; "
                       "bf16: one whole-rollout launch (a CTA per 8x16, 8x8 or 8x4 patch), bf16_per_kernel: one graph"}

    def timed(x0, T):
        x = x0.clone()
        for _ in range(3):                      # capture / first launch + warm-up
            x.copy_(x0)
            wm.wm_latent_rollout(ctx, x, T)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            x.copy_(x0)
            wm.wm_latent_rollout(ctx, x, T)
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps, x

    try:
        finals = {}
        for prec, name, fused in ((wm.WM_PREC_BF16, "bf16", 1), (wm.WM_PREC_BF16, "bf16_per_kernel", 0),
                                  (wm.WM_PREC_FP32, "fp32", 1)):
            wm.wm_set_precision(ctx, prec)
            wm.wm_set_fused_rollout(fused)
            for T in (336, 337):
                ms, x = timed(x1, T)
                res[f"{name}_T{T}_forecasts_per_s"] = 1e3 / ms
                finals[(name, T)] = x.clone()
            if name != "fp32":
                ms, _ = timed(x4, 336)
                res[f"{name}_batch4_T336_forecasts_per_s"] = 4e3 / ms
        for T in (336, 337):
            res[f"bf16_vs_fp32_final_rel_l2_T{T}"] = wm.wm_rel_l2(finals[("bf16", T)], finals[("fp32", T)])
            res[f"bf16_vs_bf16_per_kernel_final_rel_l2_T{T}"] = wm.wm_rel_l2(finals[("bf16", T)],
                                                                              finals[("bf16_per_kernel", T)])
    finally:
        wm.wm_set_fused_rollout(1)
        wm.wm_destroy(ctx)
    return res


def batch_bench(wm, torch, dev, reps=3):
    """Eight small latents with uneven leads advanced together (wm_rollout_batch,
    one captured graph): forecasts/s per precision and each lead's error
    against the FP32 plain path."""
    s = synth.SMALL
    leads = [1, 6, 7, 24, 72, 120, 240, 336]
    p6, p1 = synth.processor_weights(s, seed=0)
    x0 = [torch.from_numpy(synth.latent(s, 1, seed=1 + i)).to(dev) for i in range(len(leads))]
    ctx = wm.wm_create_from_host(wm.make_config(s, wm.WM_PREC_BF16, max_batch=len(leads)),
                                 synth.pack_weights(p6, p1))
    res = {"workload": "8 latents 4x24x48x128, leads {1,6,7,24,72,120,240,336} h, 1080 blocks; "
                       "bf16: whole-rollout launches of up to four latents, rollouts cut at steps, "
                       "fp8mlp / fp32: one graph of batched steps"}
    outs = {}
    try:
        for prec, name in ((wm.WM_PREC_BF16_FP8MLP, "fp8mlp"), (wm.WM_PREC_BF16, "bf16"), (wm.WM_PREC_FP32, "fp32")):
            wm.wm_set_precision(ctx, prec)
            lat = [x.clone() for x in x0]
            wm.wm_rollout_batch(ctx, lat, leads)        # capture + first replay
            torch.cuda.synchronize()
            total = 0.0
            for _ in range(reps):
                for a, b in zip(lat, x0):
                    a.copy_(b)
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                wm.wm_rollout_batch(ctx, lat, leads)
                e1.record()
                torch.cuda.synchronize()
                total += e0.elapsed_time(e1)
            res[f"{name}_forecasts_per_s"] = len(leads) * reps / (total / 1e3)
            outs[name] = [t.clone() for t in lat]
        for name in ("fp8mlp", "bf16"):
            res[f"{name}_vs_fp32_rel_l2_by_lead"] = {str(t): wm.wm_rel_l2(a, b)
                                                     for t, a, b in zip(leads, outs[name], outs["fp32"])}
    finally:
        wm.wm_destroy(ctx)
    return res


def hourly_ensemble_bench(wm, torch, dev, full_members=8, reps=2):
    """Hourly outputs to 14 days from one state (small latent), and ensembles:
    8 full-size members through one six-hour step, 64 small members through
    the 14-day rollout, each as one batched rollout."""
    res = {}
    s = synth.SMALL
    p6, p1 = synth.processor_weights(s, seed=0)
    ctx = wm.wm_create_from_host(wm.make_config(s, wm.WM_PREC_BF16, max_batch=64), synth.pack_weights(p6, p1))
    try:
        x = torch.from_numpy(synth.latent(s, 1, seed=1)).to(dev)
        out = torch.empty((337,) + tuple(x.shape[1:]), device=dev)
        wm.wm_rollout_hourly(ctx, x, 336, out, 16)            # capture + first replay
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            wm.wm_rollout_hourly(ctx, x, 336, out, 16)
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / reps
        res["hourly_small_14d"] = {"workload": "337 hourly latents 0..336 h from one 4x24x48x128 state, "
                                               "56 six-hour anchors + 280 batched one-hour steps",
                                   "ms_per_forecast_set": ms, "forecast_sets_per_s": 1e3 / ms}
        ens = torch.from_numpy(synth.latent(s, 64, seed=100)).to(dev)
        work = ens.clone()
        wm.wm_latent_rollout(ctx, work, 336)
        torch.cuda.synchronize()
        e0.record()
        for _ in range(reps):
            work.copy_(ens)
            wm.wm_latent_rollout(ctx, work, 336)
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / reps
        res["ensemble_small_14d"] = {"workload": "64 members 4x24x48x128, 336 h each, "
                                                 "16 whole-rollout launches of 4 members",
                                     "member_forecasts_per_s": 64e3 / ms}
    finally:
        wm.wm_destroy(ctx)
    f = synth.FULL
    p6, p1 = synth.processor_weights(f, seed=0)
    ctx = wm.wm_create_from_host(wm.make_config(f, wm.WM_PREC_BF16, max_batch=full_members),
                                 synth.pack_weights(p6, p1))
    try:
        ens = torch.from_numpy(synth.latent(f, full_members, seed=100)).to(dev)
        wm.wm_processor_step(ctx, ens, wm.WM_P6)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            wm.wm_processor_step(ctx, ens, wm.WM_P6)
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / reps
        res["ensemble_full_6h"] = {"workload": f"{full_members} members 9x90x180x768, one six-hour step as one batch",
                                   "ms_per_step": ms, "member_forecasts_per_s": full_members * 1e3 / ms}
    finally:
        wm.wm_destroy(ctx)
    return res


def serve_bench(wm, torch, n_requests=2000, rate=4.0, seed=0, bf16_only=False, n_other=120):
    """Poisson request stream on the small latent through the continuous-batching server.

    Requests: exponential inter-arrivals (mean 1/rate s), lead times uniform in
    1..336 h, latent i seeded by its request index (generated when the request
    is first needed). BF16 serves the whole stream (n_requests, 2,000 by
    default: about 500 s in real time); FP8-MLP and the FP32 plain path serve
    its first n_other requests. Reported per precision: p50/p99 latency
    (submit -> finished) at the offered rate, most requests resident at once,
    the largest batched step and how many steps advanced two or more requests
    together, and forecasts/s closed-loop at saturation (the first 480 BF16
    requests submitted at once; the others: 64). For BF16 also the first 240 requests
    under an HBM budget of one resident request (later arrivals queue until
    the slot frees); the BF16 and FP8-MLP results' error against FP32 on the
    requests all three served.
    """
    s = synth.SMALL
    p6, p1 = synth.processor_weights(s, seed=0)
    rng = np.random.default_rng(seed)
    gaps = rng.exponential(1.0 / rate, n_requests)
    leads = rng.integers(1, 337, n_requests)
    cache = {}

    def latent(i):
        if i not in cache:
            cache[i] = synth.latent(s, 1, seed=1000 + i)
        return cache[i]

    max_batch = 16
    res = {"workload": (f"Poisson arrivals {rate}/s, {n_requests} requests (BF16; FP8-MLP and FP32: the first "
                        f"{min(n_other, n_requests)}), leads U{{1..336}} h, latent 4x24x48x128, P6 8 + P1 4 blocks, "
                        f"max batch {max_batch}")}
    outs = {}

    keep = min(n_other, n_requests)   # results kept for the precision comparison
    n_sat_bf16 = min(480, n_requests)  # saturated BF16 run: these latents stay cached

    def open_loop(srv, n=n_requests):
        t0 = time.perf_counter()
        arrive = np.cumsum(gaps)
        ids, got, results = [], set(), {}
        buf = np.empty_like(latent(0))
        i = 0
        while len(got) < n:
            now = time.perf_counter() - t0
            while i < n and arrive[i] <= now:
                ids.append(wm.wm_server_submit(srv, latent(i), int(leads[i])))
                if i >= n_sat_bf16:
                    cache.pop(i, None)        # submit copied it; no later run needs it
                i += 1
            for j, rid in enumerate(ids):
                if j in got:
                    continue
                done, _ = wm.wm_server_poll(srv, rid, buf)
                if done:
                    got.add(j)
                    if j < keep:
                        results[j] = buf.copy()
            time.sleep(0.0005)
        return results, wm.wm_server_stats(srv)

    precs = ((wm.WM_PREC_BF16, "bf16"),) if bf16_only else ((wm.WM_PREC_BF16, "bf16"),
                                                            (wm.WM_PREC_BF16_FP8MLP, "fp8mlp"),
                                                            (wm.WM_PREC_FP32, "fp32"))
    for prec, name in precs:
        ctx = wm.wm_create_from_host(wm.make_config(s, prec), synth.pack_weights(p6, p1))
        lat_floats, ws = wm.wm_ctx_sizes(ctx, max_batch)
        budget = ws + (max_batch + 64) * lat_floats * 4   # 64 resident request slots
        try:
            # ---- open loop at the offered rate
            n_open = n_requests if name == "bf16" else min(n_other, n_requests)
            srv = wm.wm_server_start(ctx, budget, max_batch)
            try:
                got, st = open_loop(srv, n_open)
            finally:
                wm.wm_server_stop(srv)
            outs[name] = got
            res[f"{name}_requests"] = n_open
            res[f"{name}_p50_ms"] = st["p50_ms"]
            res[f"{name}_p99_ms"] = st["p99_ms"]
            res[f"{name}_open_loop_forecasts_per_s"] = st["forecasts_per_s"]
            res[f"{name}_max_resident"] = st["max_active"]
            res[f"{name}_max_step_batch"] = st["max_step_batch"]
            res[f"{name}_multi_request_steps"] = st["multi_request_steps"]
            if name == "bf16":
                # ---- the stream's start with room for one resident request: arrivals queue
                small = ws + (max_batch + 1) * lat_floats * 4
                n_small = min(240, max(1, n_requests // 2))
                srv = wm.wm_server_start(ctx, small, max_batch)
                try:
                    _, st = open_loop(srv, n_small)
                finally:
                    wm.wm_server_stop(srv)
                res["bf16_budget1_requests"] = n_small
                res["bf16_budget1_p50_ms"] = st["p50_ms"]
                res["bf16_budget1_p99_ms"] = st["p99_ms"]
                res["bf16_budget1_max_resident"] = st["max_active"]
                res["bf16_budget1_max_step_batch"] = st["max_step_batch"]
                res["hbm_budget_bytes"] = {"default": int(budget), "small": int(small)}
            # ---- closed loop: all requests at once, throughput at saturation
            n_sat = n_sat_bf16 if name == "bf16" else min(64, n_requests)
            srv = wm.wm_server_start(ctx, budget, max_batch)
            try:
                t0 = time.perf_counter()
                ids = [wm.wm_server_submit(srv, latent(j), int(leads[j])) for j in range(n_sat)]
                left = set(ids)
                while left:
                    for rid in list(left):
                        done, _ = wm.wm_server_poll(srv, rid, None)
                        if done:
                            left.discard(rid)
                    time.sleep(0.0005)
                dt = time.perf_counter() - t0
                sst = wm.wm_server_stats(srv)
            finally:
                wm.wm_server_stop(srv)
            res[f"{name}_saturated_forecasts_per_s"] = n_sat / dt
            res[f"{name}_saturated_requests"] = n_sat
            res[f"{name}_saturated_max_resident"] = sst["max_active"]
            res[f"{name}_saturated_max_step_batch"] = sst["max_step_batch"]
            res[f"{name}_saturated_multi_request_steps"] = sst["multi_request_steps"]
        finally:
            wm.wm_destroy(ctx)
    if bf16_only:
        return res
    common = sorted(set(outs["bf16"]) & set(outs["fp8mlp"]) & set(outs["fp32"]))
    for name in ("bf16", "fp8mlp"):
        errs = [float(np.linalg.norm(outs[name][j].astype(np.float64) - outs["fp32"][j]) /
                      np.linalg.norm(outs["fp32"][j].astype(np.float64))) for j in common]
        res[f"{name}_vs_fp32_rel_l2_median"] = float(np.median(errs))
        res[f"{name}_vs_fp32_rel_l2_max"] = float(np.max(errs))
    return res


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-fp32", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-rollout", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-serve", action="store_true")
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--no-fields", action="store_true")
    ap.add_argument("--serve-requests", type=int, default=2000)
    ap.add_argument("--serve-bf16-only", action="store_true")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
