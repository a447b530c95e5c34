#!/usr/bin/env python
"""Benchmark of the masked-block denoising path on B200.

One "step" is one whole request of the workload through the hot path: prefill of the prompt, then
block-by-block threshold decoding (denoise forwards + decisions + one finalize forward per block)
until gen_len tokens are committed.  The metric is decoded tokens per second.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--workload c2] [--impl ours|reference]

N > 1 (launched under torchrun) runs independent replicas, one per GPU, with no collective on the
data path; value = tokens of all replicas / max-over-ranks time ("weak" scaling).
`--impl reference` times the CPU oracle (oracle/) on a bounded sample of the same workload.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

# DRAM traffic (dram bytes read + written) of the dominant kernel comes from an ncu capture, kept as data in
# profiles/ncu_traffic.json (written by hand from the capture summarised next to it).  It is reported only
# while the kernel sources still hash to the value stored there; after any change to them it reads null
# until the capture is taken again.
NCU_TRAFFIC_FILE = os.path.join(ROOT, "profiles", "ncu_traffic.json")


def kernel_source_hash(files) -> str:
    import hashlib
    h = hashlib.sha256()
    for f in files:
        with open(os.path.join(ROOT, "paper_2601_07568_b200", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def ncu_traffic(kernel: str, workload: str):
    """Captured DRAM bytes of `kernel` on `workload` as {"bytes_per_layer", "bytes_fixed", "source"}, or None when
    there is no capture or the kernel has changed since."""
    try:
        with open(NCU_TRAFFIC_FILE) as f:
            data = json.load(f)
    except (OSError, ValueError):
        return None
    for e in data.get("captures", []):
        if e.get("kernel") == kernel and e.get("workload") == workload and kernel_source_hash(e.get("sources", [])) == e.get("source_hash"):
            return e
    return None


def tokens_of(w) -> int:
    return w.batch * w.gen_len


METRIC = "decoded tokens/s"
UNIT = "tokens/s"


def host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return dict(hbm_gbs=float(p["hbm_gbs"]), bf16_tflops=float(p["bf16_tflops"]),
                    bf16_tflops_sustained=float(p.get("bf16_tflops_sustained", p["bf16_tflops"])), source="measured")
    return dict(hbm_gbs=6650.0, bf16_tflops=1590.0, bf16_tflops_sustained=1400.0, source="fallback")


# ----------------------------------------------------------------------------- clocks
class ClockSampler:
    """Samples SM clock and throttle reasons with nvidia-smi while the timed region runs."""
    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
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
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for n, v in zip(names, parts[3:7]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# ----------------------------------------------------------------------------- oracle sample
_SAMPLE_WEIGHTS = {}


def oracle_sample(workload, n_denoise: int, n_finalize: int, layers=(0, 1)):
    """Time the CPU oracle, as it stands, on a bounded sample of the workload: the given layers of one
    block forward (M = block rows against a prompt-length prefix) and of one prompt forward, and the
    LM head with its statistics on one block; extrapolate to a whole request."""
    from oracle import d3_oracle as o
    from paper_2601_07568_b200 import synth_inputs as si
    shape = workload.model
    dtype = np.float64 if shape.dtype == "fp32" else np.float32
    key = (shape.name, tuple(layers))
    if key not in _SAMPLE_WEIGHTS:  # input generation is not part of the timed work
        _SAMPLE_WEIGHTS[key] = {"layers": {l: si.gen_layer(shape, l) for l in layers},
                                "lm_head": si.gen_tensor(shape, "lm_head"),
                                "tok_emb": si.gen_tensor(shape, "tok_emb", rows=(0, 8))}
    W = _SAMPLE_WEIGHTS[key]
    model = o.model_from_shape(shape, W, dtype)
    rng = np.random.default_rng(0)
    B, P = workload.block, workload.prompt_max
    kp = rng.standard_normal((P, shape.n_kv_heads, shape.d_head)).astype(dtype)
    x = rng.standard_normal((B, shape.d_model)).astype(dtype)
    xp = rng.standard_normal((P, shape.d_model)).astype(dtype)
    t0 = time.perf_counter()
    for l in layers:
        model.layer_forward(l, x, P + np.arange(B), kp, kp)
    t_layer = (time.perf_counter() - t0) / len(layers)
    t0 = time.perf_counter()
    for l in layers:
        model.layer_forward(l, xp, np.arange(P), None, None)
    t_layer_prefill = (time.perf_counter() - t0) / len(layers)
    t0 = time.perf_counter()
    lg = model.logits(x)
    o.softmax_stats(lg, shape.mask_id)
    t_head = time.perf_counter() - t0
    L = shape.n_layers
    per_seq = (n_denoise * (L * t_layer + t_head) + n_finalize * L * t_layer + L * t_layer_prefill)
    tokens_per_s = workload.gen_len / per_seq  # sequences are independent: same rate for any batch on one host
    sample = (f"layers {list(layers)} of one {B}-row block forward at prefix {P} ({t_layer * 1e3:.0f} ms/layer), of one "
              f"{P}-row prompt forward ({t_layer_prefill * 1e3:.0f} ms/layer) and the LM head + statistics on one block "
              f"({t_head * 1e3:.0f} ms); extrapolated to {L} layers and {n_denoise} denoise + {n_finalize} finalize forwards per sequence")
    return tokens_per_s, sample, dict(ms_layer=t_layer * 1e3, ms_layer_prefill=t_layer_prefill * 1e3, ms_head=t_head * 1e3)


def oracle_forward_counts(workload):
    """Forward counts of a request for the reference arm, from the oracle alone.  How many tokens a denoise
    forward commits depends on the model's logits, which only a full run of the 8B-shaped model gives; the
    method fixes the range: between one forward per block (everything clears the threshold at once) and
    one forward per token (only the forced commit each time).  The oracle's own free-running decode of the
    tiny configuration (c1, same threshold rule) gives a measured tokens-per-forward ratio, which is the
    one applied here; the two bounds are reported beside it."""
    from oracle import d3_oracle as o
    from paper_2601_07568_b200 import synth_inputs as si
    c1 = si.WORKLOADS["c1"]
    model = o.model_from_shape(c1.model, si.gen_weights(c1.model), np.float64)
    ids, lens = si.gen_prompts(c1)
    r = model.generate(ids[0, :lens[0]], c1.gen_len, c1.block, workload.threshold)
    tpf = c1.gen_len / max(r["n_denoise"], 1)
    n_blocks = workload.gen_len // workload.block
    nd = int(round(workload.gen_len / tpf))
    nd = min(max(nd, n_blocks), workload.gen_len)
    return nd, n_blocks, tpf


def run_reference(args):
    from paper_2601_07568_b200 import synth_inputs as si
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    w = si.WORKLOADS[args.workload]
    nd, nf, tpf = oracle_forward_counts(w)
    vals, sample, parts = [], "", {}
    for i in range(args.warmup + args.steps):
        v, sample, parts = oracle_sample(w, nd, nf, layers=(0,))
        if i >= args.warmup:
            vals.append(v)
    value = float(np.mean(vals))
    L = w.model.n_layers

    def rate(n_denoise):  # the same extrapolation with another forward count
        per_seq = (n_denoise * (L * parts["ms_layer"] + parts["ms_head"]) + nf * L * parts["ms_layer"] + L * parts["ms_layer_prefill"]) / 1e3
        return w.gen_len / per_seq
    sample += (f"; denoise forwards per request from the oracle's own decode of c1 at this threshold ({tpf:.2f} tokens per denoise forward); "
               f"the method allows {nf} to {w.gen_len}: {rate(nf):.2f} to {rate(w.gen_len):.2f} tokens/s")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * w.batch * w.gen_len / value,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64" if w.model.dtype == "fp32" else "f32", "data": "synthetic",
            "config": workload_config(w),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": host_cores(), "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def workload_config(w):
    return {"workload": f"{w.name}: {w.model.name}, batch {w.batch}, prompt {w.prompt_min}-{w.prompt_max}, "
                        f"generate {w.gen_len}, block {w.block}, threshold {w.threshold}",
            "l2": "inputs larger than L2 (weights read once per forward)", "replicas": "independent per GPU"}


# ----------------------------------------------------------------------------- replicas
def max_over_ranks(ms: float, dist, device) -> float:
    """The job's time is the slowest replica's: MAX all-reduce of the locally measured milliseconds
    (the only collective of a multi-GPU run; `dist` is None for one process)."""
    if dist is None:
        return float(ms)
    import torch
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_tokens_per_s(world: int, tokens_per_replica: int, steps: int, ms_max: float) -> float:
    """Independent replicas, one per GPU: every rank decodes its own copy of the workload."""
    return world * tokens_per_replica * steps / (ms_max / 1e3)


# ----------------------------------------------------------------------------- our arm
def gemm_bytes(shape, M):
    """Algorithmic bytes of each matmul launch of one M-row forward: weights + inputs + outputs."""
    d, f, V = shape.d_model, shape.d_ffn, shape.vocab
    nq, nkv = shape.n_q_heads * shape.d_head, shape.n_kv_heads * shape.d_head
    return {
        "gemm_qkv": (nq + 2 * nkv) * d * 2 + M * d * 2 + M * (nq + 2 * nkv) * 2,
        "gemm_o": d * nq * 2 + M * nq * 2 + 2 * M * d * 4,
        "gemm_gate_up": 2 * f * d * 2 + M * d * 2 + M * f * 2,
        "gemm_down": d * f * 2 + M * f * 2 + 2 * M * d * 4,
        "gemm_head": V * d * 2 + M * d * 2 + M * ((V + 127) // 128) * 16,
    }


def gemm_flops(shape, M):
    d, f, V = shape.d_model, shape.d_ffn, shape.vocab
    nq, nkv = shape.n_q_heads * shape.d_head, shape.n_kv_heads * shape.d_head
    return {"gemm_qkv": 2 * M * (nq + 2 * nkv) * d, "gemm_o": 2 * M * d * nq, "gemm_gate_up": 2 * M * 2 * f * d,
            "gemm_down": 2 * M * d * f, "gemm_head": 2 * M * V * d}


def profiled_request(ctx, w, ids_dev, lens_dev, out_dev, mode):
    """One request with an event pair around every launch of the decode loop (mode 1: every matmul a launch of its own; 2: the
    launches that the loop makes).  Returns (classes, stats, rows of all its forwards)."""
    import torch
    from paper_2601_07568_b200 import binding as d3
    d3.d3_prefill(ctx, ids_dev, lens_dev)
    torch.cuda.synchronize()
    rows0 = d3.d3_launch_count_of(ctx, "forward_rows")
    d3.d3_profile_enable(ctx, mode)
    st = d3.d3_generate(ctx, w.gen_len, w.threshold, out_dev)
    prof = d3.d3_profile_read(ctx)
    d3.d3_profile_enable(ctx, 0)
    return prof, st, d3.d3_launch_count_of(ctx, "forward_rows") - rows0


def matmul_totals(shape, prof, forwards, rows):
    """Matmul launches of a profiled request of `forwards` forwards over `rows` rows in all: (ms, launches, bytes, flops)."""
    layer_keys = ("gemm_qkv", "gemm_o", "gemm_gate_up", "gemm_down")
    keys = layer_keys + ("gemm_head", "gemm_other")
    totals = [forwards * (shape.n_layers * sum(t[k] for k in layer_keys) + t["gemm_head"])
              for t in (fn(shape, rows / max(forwards, 1)) for fn in (gemm_bytes, gemm_flops))]
    return sum(prof[k]["ms"] for k in keys), sum(prof[k]["launches"] for k in keys), *totals


def measure_batched(name, W, dev, local, world, dist, peaks, steps):
    """The batched companion workload (same model, batch 32): decoded tokens/s resident and end to end,
    ms per forward, and the tensor roofline of its matmul launches (flops / CUDA-event time / sustained peak)."""
    import torch
    from paper_2601_07568_b200 import binding as d3
    from paper_2601_07568_b200 import synth_inputs as si
    w = si.WORKLOADS[name]
    shape = w.model
    cfg = d3.make_config(shape, block=w.block, max_batch=w.batch, max_seq=w.max_seq, max_prefill_rows=w.batch * w.prompt_max)
    ctx = d3.d3_create(cfg)
    d3.d3_load_weights(ctx, d3.weights_from_numpy(shape, W), shape.n_layers)
    ids_np, lens_np = si.gen_prompts(w)
    ids_pin, lens_pin = torch.from_numpy(ids_np).pin_memory(), torch.from_numpy(lens_np).pin_memory()
    ids_dev, lens_dev = ids_pin.to(dev), lens_pin.to(dev)
    out_dev = torch.zeros((w.batch, w.gen_len), dtype=torch.int32, device=dev)
    out_pin = torch.zeros((w.batch, w.gen_len), dtype=torch.int32).pin_memory()

    def step_resident():
        d3.d3_prefill(ctx, ids_dev, lens_dev)
        return d3.d3_generate(ctx, w.gen_len, w.threshold, out_dev)

    def step_e2e():
        d3.d3_prefill(ctx, ids_pin.to(dev, non_blocking=True), lens_pin.to(dev, non_blocking=True))
        st = d3.d3_generate(ctx, w.gen_len, w.threshold, out_dev)
        out_pin.copy_(out_dev, non_blocking=True)
        torch.cuda.current_stream().synchronize()
        return st

    def timed(fn, k):
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        st = None
        for _ in range(k):
            st = fn()
        e1.record()
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()
        return max_over_ranks(e0.elapsed_time(e1), dist, dev), st

    for _ in range(3):
        step_resident()
    clocks = ClockSampler(local)
    clocks.start()
    ms_total, st = timed(step_resident, steps)
    clock_info = clocks.stop()
    ms_e2e, _ = timed(step_e2e, steps)
    ms_prefill, _ = timed(lambda: d3.d3_prefill(ctx, ids_dev, lens_dev), 3)
    ms_prefill /= 3
    prof, st_prof, rows = profiled_request(ctx, w, ids_dev, lens_dev, out_dev, 2)
    err_word = d3.d3_get_error_word(ctx)
    d3.d3_destroy(ctx)
    tokens = w.batch * w.gen_len
    gf = gemm_flops(shape, rows / max(st_prof.steps, 1))
    tot_ms, n_gemm, _, tot_flops = matmul_totals(shape, prof, st_prof.steps, rows)
    ms_step = ms_total / steps
    ms_fwd = (ms_step - ms_prefill) / max(st.steps, 1)
    layer_keys = ("gemm_qkv", "gemm_o", "gemm_gate_up", "gemm_down")
    fwd_flops = sum(gf[k] for k in layer_keys) * shape.n_layers + gf["gemm_head"]
    achieved = tot_flops / (tot_ms / 1e3) / 1e12 if tot_ms > 0 else 0.0
    return {
        "config": workload_config(w), "value": whole_job_tokens_per_s(world, tokens, steps, ms_total), "unit": UNIT,
        "value_decode_only": world * tokens / ((ms_step - ms_prefill) / 1e3), "steps": steps, "warmup": 3, "ms_per_step": ms_step,
        "e2e": {"value": whole_job_tokens_per_s(world, tokens, steps, ms_e2e), "unit": UNIT,
                "h2d_bytes_per_step": int(ids_pin.numel() * 4 + lens_pin.numel() * 4), "d2h_bytes_per_step": int(out_pin.numel() * 4)},
        "decode": {"forwards_per_request": int(st.steps), "tokens_per_denoise_forward": tokens / max(st.denoise_forwards, 1),
                   "ms_per_forward": ms_fwd, "prefill_ms": ms_prefill},
        "roofline": {"bound": "tensor", "achieved": achieved, "peak": peaks["bf16_tflops_sustained"], "unit": "TFLOP/s",
                     "frac": achieved / peaks["bf16_tflops_sustained"], "traffic": None,
                     "kernel": "gemm_pair_kernel (all matmul launches of the decode loop as it makes them, LM head included; CUDA events around every launch, which keep it from overlapping the next)",
                     "peak_source": f"of {peaks['source']} (sustained)", "launches": n_gemm, "avg_launch_us": 1e3 * tot_ms / max(n_gemm, 1),
                     "flops_per_launch": tot_flops / max(n_gemm, 1),
                     "step_effective": {"TFLOP/s": fwd_flops / (ms_fwd / 1e3) / 1e12,
                                        "frac_of_measured_tensor": fwd_flops / (ms_fwd / 1e3) / 1e12 / peaks["bf16_tflops_sustained"],
                                        "ms_per_forward": ms_fwd}},
        "clocks": clock_info, "device_error_word": err_word,
    }


def run_ours(args):
    import torch
    from paper_2601_07568_b200 import binding as d3
    from paper_2601_07568_b200 import build as d3build
    from paper_2601_07568_b200 import synth_inputs as si

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise RuntimeError("bench.py needs a CUDA device: the product path has no CPU fallback")
    torch.cuda.set_device(local)
    dev = f"cuda:{local}"
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    d3build.build()
    w = si.WORKLOADS[args.workload]
    shape = w.model
    t0 = time.time()
    W = si.gen_weights(shape)
    t_gen = time.time() - t0
    # workspace rows: the prompt forward, and the KV-refresh forward over prompt + generated blocks
    cfg = d3.make_config(shape, block=w.block, max_batch=w.batch, max_seq=w.max_seq,
                         max_prefill_rows=w.batch * w.max_seq)
    ctx = d3.d3_create(cfg)
    d3.d3_load_weights(ctx, d3.weights_from_numpy(shape, W), shape.n_layers)
    # the metric is quoted at batch 1 and 32 on the same model: the default run measures the batch-32
    # workload (c3) after the headline one, from the same host weights
    second = "c3" if (args.workload == "c2" and not args.single) else None
    if second is None:
        del W
    ids_np, lens_np = si.gen_prompts(w)
    ids_pin = torch.from_numpy(ids_np).pin_memory()
    lens_pin = torch.from_numpy(lens_np).pin_memory()
    ids_dev, lens_dev = ids_pin.to(dev), lens_pin.to(dev)
    out_dev = torch.zeros((w.batch, w.gen_len), dtype=torch.int32, device=dev)
    out_pin = torch.zeros((w.batch, w.gen_len), dtype=torch.int32).pin_memory()

    def step_resident():
        d3.d3_prefill(ctx, ids_dev, lens_dev)
        return d3.d3_generate(ctx, w.gen_len, w.threshold, out_dev)

    def step_e2e():
        a = ids_pin.to(dev, non_blocking=True)
        b = lens_pin.to(dev, non_blocking=True)
        d3.d3_prefill(ctx, a, b)
        st = d3.d3_generate(ctx, w.gen_len, w.threshold, out_dev)
        out_pin.copy_(out_dev, non_blocking=True)
        torch.cuda.current_stream().synchronize()
        return st

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    def timed(fn, k):
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        st = None
        for _ in range(k):
            st = fn()
        e1.record()
        barrier()
        return max_over_ranks(e0.elapsed_time(e1), dist, dev), st

    for _ in range(args.warmup):
        step_resident()
    clocks = ClockSampler(local)
    clocks.start()
    launches0 = d3.d3_launch_count(ctx)
    ms_total, st = timed(step_resident, args.steps)
    launches = d3.d3_launch_count(ctx) - launches0
    clock_info = clocks.stop()
    ms_e2e, _ = timed(step_e2e, args.steps)

    # the paper's multi-block decoding on the same request, beside the headline number, with as many
    # blocks in flight as 128 rows hold
    multiblock = None
    mb_window = min(8, 128 // (w.batch * w.block))  # rounds of at most 128 rows stay on the skinny kernels
    if mb_window >= 2:
        def step_multiblock():
            d3.d3_prefill(ctx, ids_dev, lens_dev)
            return d3.d3_generate_multiblock(ctx, w.gen_len, w.threshold, out_dev, mb_window)
        step_multiblock()
        ms_mb, st_mb = timed(step_multiblock, args.steps)
        multiblock = {"max_active": mb_window, "value": whole_job_tokens_per_s(world, tokens_of(w), args.steps, ms_mb), "unit": UNIT,
                      "rounds_per_request": int(st_mb.steps), "tokens_per_round": tokens_of(w) / max(int(st_mb.steps), 1),
                      "ms_per_round": ms_mb / args.steps / max(int(st_mb.steps), 1)}

    # KV-refresh: one forward over the whole stored prefix (prompt + generated blocks) of every sequence,
    # timed alone after a request, and the request decoded with a refresh after every fourth block
    ms_refresh, _ = timed(lambda: d3.d3_refresh_cache(ctx, w.batch), 3)
    ms_refresh /= 3
    refresh_rows = int(w.batch * (int(lens_np.max()) + w.gen_len))
    d3.d3_set_cache_policy(ctx, 1, 4)
    step_resident()
    ms_rf, st_rf = timed(step_resident, args.steps)
    n_refresh = d3.d3_refresh_count(ctx)
    d3.d3_set_cache_policy(ctx, 1, 0)
    kv_refresh = {"rows": refresh_rows, "ms": ms_refresh,
                  # matmul flops of the layers (no LM head in a refresh forward; attention not counted)
                  "tflops": shape.n_layers * sum(v for k, v in gemm_flops(shape, refresh_rows).items() if k != "gemm_head")
                  / (ms_refresh * 1e-3) / 1e12,
                  "decode_refresh_every_4_blocks": {"value": whole_job_tokens_per_s(world, tokens_of(w), args.steps, ms_rf), "unit": UNIT,
                                                    "refreshes_per_request": int(n_refresh)}}

    # temperature sampling (Gumbel-max in the LM-head epilogue) on the same request
    d3.d3_set_sampling(ctx, 0.1, 20260107)
    step_resident()
    ms_sm, st_sm = timed(step_resident, args.steps)
    d3.d3_set_sampling(ctx, 0.0, 0)
    sampling = {"temperature": 0.1, "value": whole_job_tokens_per_s(world, tokens_of(w), args.steps, ms_sm), "unit": UNIT,
                "forwards_per_request": int(st_sm.steps),
                "ms_per_step": ms_sm / args.steps / max(int(st_sm.steps), 1)}

    # pseudo-trajectory extraction (threshold 1: one token per forward, full length) on the same request,
    # and the noisy-sequence builder on a training-sized batch of responses
    cs_dev = torch.zeros((w.batch, w.gen_len), dtype=torch.int32, device=dev)
    def step_extract():
        d3.d3_prefill(ctx, ids_dev, lens_dev)
        return d3.d3_generate(ctx, w.gen_len, 1.0, out_dev, cs_dev)
    ms_ex, st_ex = timed(step_extract, 1)
    rank_dev = torch.zeros_like(cs_dev)
    d3.d3_trajectory_rank(ctx, cs_dev, rank_dev)
    nb, nn = 16384, w.gen_len
    gnr = torch.Generator(device=dev).manual_seed(7)
    y_big = torch.randint(0, shape.vocab - 2, (nb, nn), dtype=torch.int32, device=dev, generator=gnr)
    rank_big = rank_dev[:1].expand(nb, nn).contiguous()
    s_big = torch.randint(0, nn // 2, (nb,), dtype=torch.int32, device=dev, generator=gnr)
    k_big = torch.full((nb,), w.block, dtype=torch.int32, device=dev)
    m_big = torch.randint(0, w.block + 1, (nb,), dtype=torch.int32, device=dev, generator=gnr)
    noisy = torch.empty_like(y_big)
    d3.d3_noisy_sequence(ctx, y_big, rank_big, s_big, k_big, m_big, noisy)
    ms_ns, _ = timed(lambda: d3.d3_noisy_sequence(ctx, y_big, rank_big, s_big, k_big, m_big, noisy), 20)
    ms_ns /= 20
    trajectory = {"extraction": {"value": whole_job_tokens_per_s(world, tokens_of(w), 1, ms_ex), "unit": UNIT,
                                 "forwards_per_request": int(st_ex.denoise_forwards + st_ex.finalize_forwards) // max(w.batch, 1)},
                  "noisy_sequence": {"sequences": nb, "tokens_each": nn, "us_per_launch": ms_ns * 1e3,
                                     "GB/s": 3 * nb * nn * 4 / (ms_ns * 1e-3) / 1e9}}
    del y_big, rank_big, noisy

    # kernel times of the decode loop, events around every launch: as it makes them, and with every matmul by itself
    prof, st_prof, prof_rows = profiled_request(ctx, w, ids_dev, lens_dev, out_dev, 2)
    split, st_split, split_rows = profiled_request(ctx, w, ids_dev, lens_dev, out_dev, 1)
    # prefill alone
    ms_prefill, _ = timed(lambda: d3.d3_prefill(ctx, ids_dev, lens_dev), 3)
    ms_prefill /= 3
    err_word = d3.d3_get_error_word(ctx)
    tokens = w.batch * w.gen_len
    value = whole_job_tokens_per_s(world, tokens, args.steps, ms_total)
    e2e_value = whole_job_tokens_per_s(world, tokens, args.steps, ms_e2e)
    ms_step = ms_total / args.steps

    peaks = measured_peaks()
    gb, gf = (fn(shape, prof_rows / max(st_prof.steps, 1)) for fn in (gemm_bytes, gemm_flops))  # of a forward with the mean rows
    layer_keys = ("gemm_qkv", "gemm_o", "gemm_gate_up", "gemm_down")
    # K/V read by the attention of one forward at mid-generation
    kv_mid = 2 * shape.n_layers * shape.n_kv_heads * shape.d_head * 2 * sum(int(l) + w.gen_len // 2 for l in lens_np)
    tot_ms, n_dom, tot_bytes, tot_flops = matmul_totals(shape, prof, st_prof.steps, prof_rows)
    dominant = ("gemm_sk_kernel (O-proj, gate/up, down and the next layer's QKV or the LM head in a launch) and the other matmul launches of "
                "the decode loop as it makes them; CUDA events around every launch, which keep it from overlapping the next")
    hbm_bound = tot_flops / max(tot_bytes, 1) < peaks["bf16_tflops_sustained"] * 1e12 / (peaks["hbm_gbs"] * 1e9)
    if hbm_bound:
        achieved = tot_bytes / (tot_ms / 1e3) / 1e9 if tot_ms > 0 else 0.0
        roofline = {"bound": "hbm", "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                    "frac": achieved / peaks["hbm_gbs"], "traffic": None,
                    "frac_of_8TBs_nominal": achieved / 8000.0}
    else:
        achieved = tot_flops / (tot_ms / 1e3) / 1e12 if tot_ms > 0 else 0.0
        roofline = {"bound": "tensor", "achieved": achieved, "peak": peaks["bf16_tflops_sustained"], "unit": "TFLOP/s",
                    "frac": achieved / peaks["bf16_tflops_sustained"], "traffic": None}
    # whole forward as one unit: weights + KV of one forward over its share of the timed region
    ms_fwd = (ms_step - ms_prefill) / max(st.steps, 1)
    fwd_bytes = sum(gb[k] for k in layer_keys) * shape.n_layers + gb["gemm_head"] + kv_mid
    fwd_flops = sum(gf[k] for k in layer_keys) * shape.n_layers + gf["gemm_head"]
    roofline["step_effective"] = {"GB/s": fwd_bytes / (ms_fwd / 1e3) / 1e9, "TFLOP/s": fwd_flops / (ms_fwd / 1e3) / 1e12,
                                  "frac_of_measured_hbm": fwd_bytes / (ms_fwd / 1e3) / 1e9 / peaks["hbm_gbs"],
                                  "frac_of_8TBs_nominal": fwd_bytes / (ms_fwd / 1e3) / 1e9 / 8000.0,
                                  "frac_of_measured_tensor": fwd_flops / (ms_fwd / 1e3) / 1e12 / peaks["bf16_tflops_sustained"],
                                  "ms_per_forward": ms_fwd, "bytes_per_forward": fwd_bytes}
    cap = ncu_traffic("gemm_sk_kernel", w.name) if hbm_bound else None
    if cap is not None and n_dom > 0:
        # the capture ran the model cut to a few layers: a forward's traffic and launches grow in proportion to them; per launch
        per_forward = float(cap["bytes_per_layer"]) * shape.n_layers + float(cap.get("bytes_fixed", 0.0))
        roofline["traffic"] = per_forward / (float(cap.get("launches_per_layer", 0)) * shape.n_layers + float(cap.get("launches_fixed", 1)))
        roofline["traffic_source"] = cap.get("source", "ncu")
    roofline.update({"kernel": dominant, "peak_source": f"of {peaks['source']}",
                     "launches": n_dom, "avg_launch_us": 1e3 * tot_ms / max(n_dom, 1),
                     "algorithmic_bytes_per_launch": tot_bytes / max(n_dom, 1)})
    # (the split schedule: what a matmul takes by itself, not what the decode loop runs)
    per_class = {"schedule": "every matmul a launch of its own"}
    gbs, gfs = (fn(shape, split_rows / max(st_split.steps, 1)) for fn in (gemm_bytes, gemm_flops))
    for k, v in split.items():
        if v["launches"] == 0:
            continue
        e = {"ms": round(v["ms"], 3), "launches": v["launches"], "us_per_launch": round(1e3 * v["ms"] / v["launches"], 2)}
        if k in gbs and v["ms"] > 0:
            e["GB/s"] = round(gbs[k] * v["launches"] / (v["ms"] / 1e3) / 1e9, 1)
            e["TFLOP/s"] = round(gfs[k] * v["launches"] / (v["ms"] / 1e3) / 1e12, 1)
        per_class[k] = e
    forwards = st.steps
    line = {
        "metric": METRIC, "value": value, "value_decode_only": world * tokens / ((ms_step - ms_prefill) / 1e3),
        "value_note": "value: whole requests, prefill inside the timed region; value_decode_only: the decode loop alone (prefill timed separately)",
        "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16" if shape.dtype == "bf16" else "f32",
        "data": "synthetic", "config": workload_config(w),
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": int(ids_pin.numel() * 4 + lens_pin.numel() * 4),
                "d2h_bytes_per_step": int(out_pin.numel() * 4)},
        "gpu_launches": int(launches), "clocks": clock_info, "roofline": roofline,
        "decode": {"forwards_per_request": int(forwards), "denoise_forwards": int(st.denoise_forwards),
                   "finalize_forwards": int(st.finalize_forwards), "tokens_per_denoise_forward": tokens / max(st.denoise_forwards, 1),
                   "tokens_per_forward_incl_finalize": tokens / max(st.denoise_forwards + st.finalize_forwards, 1),
                   "ms_per_forward": (ms_step - ms_prefill) / max(forwards, 1), "prefill_ms": ms_prefill,
                   "forced_commits": int(st.forced_commits)},
        "multiblock": multiblock, "kv_refresh": kv_refresh, "trajectory": trajectory, "sampling": sampling, "kernels": per_class, "device_error_word": err_word, "weight_gen_s": round(t_gen, 1),
        "device_bytes": d3.d3_device_bytes(ctx),
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        nd = int(st.denoise_forwards // w.batch)
        nf = int(st.finalize_forwards // w.batch)
        v, sample, _ = oracle_sample(w, nd, nf)
        line["cpu_baseline"] = {"value": v, "unit": UNIT, "cores": host_cores(), "kind": "oracle", "sample": sample}
    d3.d3_destroy(ctx)
    if second is not None:
        torch.cuda.empty_cache()
        line["workloads"] = {second: measure_batched(second, W, dev, local, world, dist, peaks, max(3, min(args.steps, 5)))}
        del W
    if rank == 0:
        print(json.dumps(line))
    if dist is not None:
        dist.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--workload", default="c2", choices=["c1", "c2", "c3", "c4", "c5"])
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--single", action="store_true", help="only the named workload (no batch-32 companion of c2)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
