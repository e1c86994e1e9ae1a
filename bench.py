#!/usr/bin/env python
"""ProxyFormer layer forward + backward throughput on GB300.

Workload: one causal 1D layer of the 12-layer long-context stack at the P = 64
position: L = 262144 tokens, d = 1024, 16 heads x 64, two-level 8 x 8
compression, gated injection, bf16 with fp32 accumulation, batch 1 per GPU.
A step is proxy_layer_fwd + proxy_layer_bwd over that sequence (inputs already
resident in HBM); `value` is tokens per second over all ranks.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

--impl reference times the float64 CPU oracle on the host cores instead (a
bounded slice of the same workload per step); it is a deliberately slow
baseline, not a GPU implementation.  Prints one JSON line (rank 0).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
METRIC = "ProxyFormer layer fwd+bwd tokens/s at L=256K, P=64; % of GB300 roofline"
UNIT = "tokens/s"
WORKLOAD = "proxyformer_layer_causal1d_L262144_d1024_h16x64_P64_8x8_gated_bf16_fwd_bwd"
SAMPLE_L = 2048       # tokens of one reference-arm step (32 proxies)
CPU_SLICE_L = 65536   # tokens of the cpu_baseline slice (1024 proxies)
PEAKS_FALLBACK = {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=("ours", "reference"), default="ours")
    ap.add_argument("--e2e-steps", type=int, default=10)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-decode", action="store_true")
    ap.add_argument("--no-configs", action="store_true",
                    help="skip the other workloads (fp32 layer, L=65536 layer, 2D layer, stack)")
    ap.add_argument("--decode-steps", type=int, default=128)
    ap.add_argument("--case", default="",
                    choices=("", "layer", "c1", "c2", "c5", "cross", "lm_history", "decode"),
                    help="profiling helper: run only this workload's step (--batch / --L shrink "
                         "it) and print its time; not the benchmark line")
    ap.add_argument("--batch", type=int, default=0, help="batch of --case (default: its own)")
    ap.add_argument("--detail", default="",
                    help="also write the per-kernel breakdowns of every workload to this JSON file")
    ap.add_argument("--L", type=int, default=0,
                    help="tokens per sequence (default: the workload's 262144; smaller values "
                         "are for profiling captures only)")
    return ap.parse_args()


def host_cores() -> int:
    return int(os.environ.get("OPENBLAS_NUM_THREADS") or os.cpu_count() or 1)


def workload_spec(L: int = 0):
    import dataclasses

    import pf_synth as S
    spec = S.spec_c3_layer(64)
    return dataclasses.replace(spec, L=L) if L else spec


def config_dict(spec, extra=None):
    name = WORKLOAD if spec.L == 262144 else WORKLOAD.replace("L262144", f"L{spec.L}")
    c = {"workload": name, "batch_per_gpu": spec.batch, "L": spec.L, "d": spec.d,
         "heads": spec.n_heads, "head_dim": spec.dh, "P": spec.P, "levels": spec.levels,
         "k1": spec.k1, "k2": spec.k2, "mode": "causal_1d", "inject": "gated",
         "l2": "inputs larger than L2 (X, dX_out, X_out, dX are 512 MiB each; L2 is 129 MB)"}
    c.update(extra or {})
    return c


# ------------------------------------------------------------------ oracle leg
def oracle_sample_seconds(L_s: int, reps: int = 1):
    """Wall seconds of one oracle fwd+bwd over an L_s-token slice of the workload."""
    import numpy as np
    import pf_synth as S
    from oracle import layer as OL
    full = workload_spec()
    spec = S.LayerSpec(batch=1, L=L_s, d=full.d, n_heads=full.n_heads, P=full.P,
                       levels=full.levels, k1=full.k1, k2=full.k2)
    inp = S.make_layer_inputs(spec, 2)
    times = []
    for _ in range(reps):
        t0 = time.perf_counter()
        OL.layer_fwd(spec, inp, inp["X"])
        OL.layer_bwd(spec, inp, inp["X"], inp["G"], None, None, inp["dH_out"])
        times.append(time.perf_counter() - t0)
    return times


def cpu_baseline_subprocess():
    """Run the oracle slice in a fresh interpreter with an explicit BLAS thread count."""
    cores = os.cpu_count() or 1
    env = dict(os.environ, OPENBLAS_NUM_THREADS=str(cores), OMP_NUM_THREADS=str(cores))
    code = ("import json, bench; t = bench.oracle_sample_seconds(%d, 1); print(json.dumps(t))"
            % CPU_SLICE_L)
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=900)
    if r.returncode != 0:
        return {"value": None, "unit": UNIT, "cores": cores, "kind": "oracle",
                "sample": "failed: " + r.stderr.strip().splitlines()[-1][:200]}
    t = json.loads(r.stdout.strip().splitlines()[-1])
    return {"value": CPU_SLICE_L / min(t), "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"one fwd+bwd of the float64 oracle over a {CPU_SLICE_L}-token slice "
                      f"({CPU_SLICE_L // 64} proxies) of the same layer shape, {min(t):.1f} s"}


# ------------------------------------------------------------ ranks (N > 1)
def rank_seed(rank: int) -> int:
    """Input seed of a rank: every replica draws its own batch (weak scaling)."""
    return 2 + 1000 * rank


def max_over_ranks(x: float, world: int, device: str = "cuda") -> float:
    """The slowest rank's time: all_reduce(MAX) over the process group."""
    if world <= 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(tokens_per_rank: float, world: int, ms: float) -> float:
    """Whole-job tokens/s: every rank's tokens over the slowest rank's step."""
    return tokens_per_rank * world / (ms / 1e3)


def run_reference(args, rank: int):
    if rank != 0:
        return
    cores = host_cores()
    spec = workload_spec()
    times = []
    for i in range(args.warmup + args.steps):
        t = oracle_sample_seconds(SAMPLE_L, 1)[0]
        if i >= args.warmup:
            times.append(t)
    sec = statistics.mean(times)
    value = SAMPLE_L / sec
    line = {"metric": METRIC, "value": value, "unit": UNIT, "impl": "reference",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": sec * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": config_dict(spec, {"oracle_slice_tokens": SAMPLE_L}),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": f"each step: float64 oracle fwd+bwd over a {SAMPLE_L}-token "
                                       f"slice of the workload"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ------------------------------------------------------------------ clocks
class ClockSampler:
    """nvidia-smi samples (every 50 ms) taken while the timed region runs."""
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_id: str):
        self.rows = []
        self.t0 = self.t1 = None
        try:
            self.p = subprocess.Popen(["nvidia-smi", "-i", gpu_id, "--query-gpu=" + self.FIELDS,
                                       "--format=csv,noheader,nounits", "-lms", "50"],
                                      stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.p = None
            return
        self.th = threading.Thread(target=self._read, daemon=True)
        self.th.start()

    def _read(self):
        for line in self.p.stdout:
            self.rows.append((time.time(), [x.strip() for x in line.split(",")]))

    def mark(self, start: bool):
        if start:
            self.t0 = time.time()
        else:
            self.t1 = time.time()

    def window(self, t0, t1):
        """Median SM clock, maximum clock and active throttle reasons of the
        samples taken between wall times t0 and t1."""
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        rows = [r for t, r in list(self.rows) if t0 - 0.06 <= t <= t1]
        sm, mx, reasons = [], [], set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        for r in rows:
            try:
                sm.append(float(r[0]))
                mx.append(float(r[1]))
            except (ValueError, IndexError):
                continue
            for n, v in zip(names, r[4:8]):
                if v.strip().lower() == "active":
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": sorted(reasons),
                "samples": len(sm)}

    def stop(self):
        """Ends sampling; the statistics of the window marked by mark()."""
        if self.p is None:
            return self.window(0, 0)
        time.sleep(0.12)
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.p.kill()
        return self.window(self.t0 or 0, self.t1 or 0)


def gpu_smi_id(torch, dev: int) -> str:
    try:
        u = str(torch.cuda.get_device_properties(dev).uuid)
        return u if u.startswith("GPU-") else "GPU-" + u
    except Exception:
        vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
        return vis.split(",")[dev] if vis else str(dev)


# ------------------------------------------------------------------ our leg
def kernel_files(label: str):
    """Source files that define the kernel behind a timing label."""
    if label == "attn_fwd":
        return ["attention_tc.cu", "common.cuh"]
    if label.startswith("attn_"):
        return ["attention_bwd_tc.cu", "attention.cu", "common.cuh"]
    if label.startswith("decode_"):
        return ["decode.cu", "common.cuh"]
    if label.startswith(("inj_bwd", "colsum", "pad_rows")):
        return ["elementwise.cu", "common.cuh"]
    return ["gemm_tc.cuh", "gemm.cu", "common.cuh"]


def source_hash(label: str) -> str:
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2608_23463_gb300", "csrc")
    for f in kernel_files(label):
        with open(os.path.join(csrc, f), "rb") as fh:
            h.update(f.encode() + fh.read())
    return h.hexdigest()[:16]


def traffic_from_profile(label: str, units: float):
    """DRAM bytes per launch of `label` from profiles/traffic.txt, whose lines
    read: label dram_bytes_per_launch units_captured kernel_source_hash.  The
    captured bytes are scaled to this launch by units (tokens); None when the
    kernel has no capture or its source changed since."""
    path = os.path.join(ROOT, "profiles", "traffic.txt")
    if not os.path.exists(path):
        return None
    for line in open(path):
        parts = line.split()
        if len(parts) >= 4 and not line.startswith("#") and parts[0] == label:
            if parts[3] != source_hash(label):
                return None
            return float(parts[1]) * units / float(parts[2])
    return None


def measure_decode(torch, pf, S, steps: int):
    """Proxy-KV decode step at the paper's decode shape: B = 8, d = 2048, 16 x 128
    heads, 16384 cached proxies per sequence, open block cycling through 0..63
    tokens.  Each step is timed with CUDA events on its stream; the open block
    is reset between passes outside the timed spans."""
    import numpy as np

    from paper_2608_23463_gb300.decode import ProxyKVCache
    spec = S.spec_c4()
    prm = S.make_decode_params(spec, 3)
    st = S.make_decode_state(spec, 3, [spec.capacity] * spec.batch, [0] * spec.batch)
    cache = ProxyKVCache(spec, prm, st)
    del st
    x = torch.from_numpy(S.round_bf16(np.random.default_rng(4).standard_normal(
        (spec.batch, spec.d)).astype(np.float32))).cuda().to(torch.bfloat16)
    y = torch.empty_like(x)
    stream = torch.cuda.current_stream()
    for _ in range(3):
        cache.step(x, y)
    cache.s["n_open"].zero_()
    torch.cuda.synchronize()
    def run(timing: bool):
        pairs = []
        cache.s["n_open"].zero_()
        pf.pf_timing_enable(timing)
        for i in range(steps):
            if i and i % spec.P == 0:
                cache.s["n_open"].zero_()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            cache.step(x, y)
            e1.record(stream)
            pairs.append((e0, e1))
        torch.cuda.synchronize()
        pf.pf_sync_check(stream.cuda_stream)
        kern = {k: v["ms"] / steps for k, v in pf.pf_timing_collect().items()} if timing else {}
        pf.pf_timing_enable(False)
        return sum(a.elapsed_time(b) for a, b in pairs) / steps, kern

    ms_direct, _ = run(False)  # one C-ABI call per step, no per-launch events
    _, kern = run(True)  # per-kernel breakdown (events around every launch)
    # the step time: the step's four launches captured once as a CUDA graph and
    # replayed back to back, P steps (one open block) per timed span
    graph = cache.capture_step(x, y)
    total, done = 0.0, 0
    while done < steps:
        n = min(spec.P, steps - done)
        cache.s["n_open"].zero_()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(n):
            graph.replay()
        e1.record(stream)
        torch.cuda.synchronize()
        total += e0.elapsed_time(e1)
        done += n
    pf.pf_sync_check(stream.cuda_stream)
    ms = total / steps
    # one block-triggered append (full open blocks, one free cache row each)
    cache.s["n_open"].fill_(spec.P)
    cache.s["n_proxy"].fill_(spec.capacity - 1)
    cache.append()
    cache.s["n_open"].fill_(spec.P)
    cache.s["n_proxy"].fill_(spec.capacity - 1)
    torch.cuda.synchronize()
    a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a0.record(stream)
    cache.append()
    a1.record(stream)
    torch.cuda.synchronize()
    pf.pf_sync_check(stream.cuda_stream)
    return spec, ms, ms_direct, a0.elapsed_time(a1), decode_step_bytes(spec, steps), kern


def decode_step_bytes(spec, steps: int) -> float:
    """Algorithmic HBM bytes of one decode step (Sec. 3.8), bf16: the K and V
    rows of every cached proxy of every sequence, the weights read once
    (W_qkv, W_o, the alpha MLP's first layer d x d/8), the open block's K and
    V rows (on average half full over the timed steps), the token in and the
    output out."""
    B, d, cap = spec.batch, spec.d, spec.capacity
    mean_open = (min(steps, spec.P) + 1) / 2.0
    return (2 * B * cap * d * 2 + (3 * d * d + d * d + d * d // 8) * 2
            + B * mean_open * 2 * d * 2 + 2 * B * d * 2)


def timed_steps(torch, pf, fn, steps: int, warmup: int):
    """Mean ms per call of fn (CUDA events on the current stream), the wall
    times bracketing the timed calls (for the clock samples), and the
    library's per-launch records: FLOPs and bytes per call as the kernels
    count them, and the label with the largest time."""
    stream = torch.cuda.current_stream()
    for _ in range(warmup):
        fn()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    w0 = time.time()
    e0.record(stream)
    for _ in range(steps):
        fn()
    e1.record(stream)
    torch.cuda.synchronize()
    w1 = time.time()
    ms = e0.elapsed_time(e1) / steps
    pf.pf_sync_check(stream.cuda_stream)
    pf.pf_timing_enable(True)  # breakdown pass
    for _ in range(steps):
        fn()
    torch.cuda.synchronize()
    t = pf.pf_timing_collect()
    pf.pf_timing_enable(False)
    pf.pf_sync_check(stream.cuda_stream)
    flops = sum(v["flops"] * v["launches"] for v in t.values()) / steps
    nbytes = sum(v["bytes"] * v["launches"] for v in t.values()) / steps
    total = sum(v["ms"] for v in t.values()) or 1.0
    dom, dv = max(t.items(), key=lambda kv: kv[1]["ms"])
    top = sorted(t.items(), key=lambda kv: -kv[1]["ms"])[:8]
    return ms, (flops, nbytes), {"kernel": dom, "share": dv["ms"] / total,
                                 "kernels_ms_per_step": {k: v["ms"] / steps for k, v in top},
                                 "launches_per_step": sum(v["launches"] for v in t.values())
                                 / steps}, (w0, w1)


# ------------------------------------------------------- algorithmic work
def layer_work(spec, train: bool = True):
    """Algorithmic FLOPs and HBM bytes of one layer step (forward, plus the
    backward when `train`), from the method's own operation counts (Eq.
    complexity, Sec. 4), not from what the kernels happen to move.

    FLOPs, per sequence (m = ceil(L/P) proxies, tokens df wide, proxies d):
      compression 2 m P df d (level 1) + 2 m k2 d d (level 2);
      decompression the mirror image, w = df (2 df for affine injection);
      proxy attention 8 m d^2 (Q, K, V, O) + 4 d per visible (query, key)
      pair (m(m+1)/2 causal, m^2 bidirectional); the MLP interaction
      16 m d^2; the cross injection 2 L df (d + heads) + 4 m d^2 + 4 d per
      visible (token, proxy) pair + 2 L d df instead of the decompression.
      The backward costs twice the linear terms and 2.5 times the attention.
    Bytes: the forward reads X twice (compression, injection) and writes
    X_out; the backward reads dX_out and X and writes dX; every weight is
    read once per pass and its fp32 gradient written once."""
    B, L, d, df, P = spec.batch, spec.L, spec.d, spec.df, spec.P
    m = -(-L // P)
    nh = spec.n_heads
    k2 = spec.k2 if spec.levels == 2 else 1
    elt = 2 if spec.dtype == 1 else 4
    affine = spec.inject == 2
    cross = spec.inject == 3
    w_tok = 2 * df if affine else df
    lin = 2.0 * m * P * df * d + (2.0 * m * k2 * d * d if spec.levels == 2 else 0.0)
    wts = P // k2 * df * d + (k2 * d * d if spec.levels == 2 else 0)
    if cross:
        vis_x = (P * m * (m - 1) / 2.0) if spec.mode == 0 else float(L) * m
        lin += 2.0 * L * df * (d + nh) + 4.0 * m * d * d + 2.0 * L * d * df
        wts += df * (d + nh) + 2 * d * d + d * df
        att_x = 4.0 * d * vis_x
    else:
        lin += 2.0 * m * k2 * d * (P // k2) * w_tok + (2.0 * m * d * k2 * d if spec.levels == 2
                                                        else 0.0)
        wts += d * (P // k2) * w_tok + (d * k2 * d if spec.levels == 2 else 0)
        att_x = 0.0
    interact = getattr(spec, "interact", 0)
    att = 0.0
    if interact == 0:
        lin += 8.0 * m * d * d
        wts += 4 * d * d
        vis = m * (m + 1) / 2.0 if spec.mode == 0 else float(m) * m
        att = 4.0 * d * vis
    elif interact == 2:
        lin += 16.0 * m * d * d
        wts += 8 * d * d
    fwd_flops = B * (lin + att + att_x)
    act = B * L * df * elt
    flops = fwd_flops
    nbytes = 3.0 * act + wts * elt
    if train:
        flops += B * (2.0 * lin + 2.5 * (att + att_x))
        nbytes += 3.0 * act + wts * elt + 4.0 * wts
    return flops, nbytes


def segments_work(d, nh, levels, segs):
    """``layer_work`` of a layer with temporal-distance ratios: each segment's
    compression and decompression at its own ratio, one causal attention over
    all the proxies, weights of every segment."""
    import pf_synth as S
    flops = nbytes = 0.0
    m_tot = 0
    for sg in segs:
        kw = dict(k1=sg[2], k2=sg[3]) if levels == 2 else {}
        sp = S.LayerSpec(batch=1, L=sg[0], d=d, n_heads=nh, P=sg[1], levels=levels,
                         interact=S.F_IDENTITY, **kw)
        f, b = layer_work(sp)
        flops += f
        nbytes += b
        m_tot += -(-sg[0] // sg[1])
    att = 4.0 * d * m_tot * (m_tot + 1) / 2.0
    flops += 8.0 * m_tot * d * d * 3 + 3.5 * att
    nbytes += 4 * d * d * 8
    return flops, nbytes


def compute_peak(peaks, clocks):
    """bf16 dense peak for a kernel timed at the sampled SM clock: the burst
    figure (measured at the maximum clock) scaled by median / maximum clock,
    never above the burst figure."""
    burst = peaks["bf16_tflops"]
    mhz, mx = (clocks or {}).get("sm_mhz"), (clocks or {}).get("sm_max_mhz")
    if mhz and mx:
        return burst * min(1.0, mhz / mx), f"bf16_tflops (burst) x {mhz:.0f}/{mx:.0f} MHz"
    return burst, "bf16_tflops (burst; no clock samples)"


def measure_ffma_peak(torch, pf):
    """The fp32 FMA pipe's peak, measured with the library's probe kernel
    (CUDA events, best of 5): TFLOP/s."""
    blocks, iters = 8 * 152, 4096
    out = torch.empty(blocks * 512, dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream()
    pf.pf_probe_ffma(out, blocks, iters, stream.cuda_stream)
    torch.cuda.synchronize()
    best = float("inf")
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        pf.pf_probe_ffma(out, blocks, iters, stream.cuda_stream)
        e1.record(stream)
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return 2.0 * blocks * 512 * 8 * iters / (best / 1e3) / 1e12


def config_entry(metric, tokens, ms, work, dom, peaks, steps, clocks=None, ffma=None,
                 rec=None):
    """One workload's line: throughput and its roofline fraction, the bound
    being the larger of algorithmic FLOPs at the compute peak (bf16 tensor, or
    the measured FFMA peak for fp32) and algorithmic bytes at HBM bandwidth."""
    flops, nbytes = work
    if ffma:
        comp_peak, src = ffma, "fp32 FFMA, measured by the probe kernel"
    else:
        comp_peak, src = compute_peak(peaks, clocks)
    t_c = flops / (comp_peak * 1e12) * 1e3
    t_b = nbytes / (peaks["hbm_gbs"] * 1e9) * 1e3
    roof_ms = max(t_c, t_b)
    bound = ("alu" if ffma else "tensor") if t_c >= t_b else "hbm"
    e = {"metric": metric, "value": tokens / (ms / 1e3), "unit": "tokens/s",
         "ms_per_step": ms, "steps": steps,
         "roofline": {"bound": bound, "flops_per_step": flops, "bytes_per_step": nbytes,
                      "compute_peak_tflops": comp_peak, "compute_peak_source": src,
                      "roofline_ms": roof_ms, "frac": roof_ms / ms, **dom}}
    if rec:
        e["roofline"]["flops_per_step_kernel_records"] = rec[0]
    if clocks:
        e["clocks"] = clocks
    return e


def measure_configs(torch, pf, S, peaks, warmup: int, sampler=None, ffma=None):
    """The other paper workloads, each timed on its own (fresh buffers); the
    clock samples of each one's timed window set its compute peak."""
    from paper_2608_23463_gb300.layer import ProxyLayer, to_device
    from paper_2608_23463_gb300.stack import ProxyStack
    out = {}

    def clk(win):
        return sampler.window(*win) if sampler else None

    def layer_case(spec, seed, train, steps):
        inp = S.make_layer_inputs(spec, seed, with_grads=train)
        dt = torch.bfloat16 if spec.dtype == S.BF16 else torch.float32
        lay = ProxyLayer(spec, inp)
        X = to_device(inp["X"], dt)
        G = to_device(inp["G"], dt) if train else None
        t = to_device(inp["t"], torch.float32) if "t" in inp else None
        del inp
        Xo, dX = lay.empty_act(), lay.empty_act()

        def step():
            lay.forward(X, None, t, X_out=Xo, train=train)
            if train:
                lay.backward(X, G, None, t, dX=dX)
        return timed_steps(torch, pf, step, steps, warmup)

    def entry(key, metric, spec, seed, train, steps, **kw):
        ms, rec, dom, win = layer_case(spec, seed, train, steps)
        out[key] = config_entry(metric, spec.batch * spec.L, ms, layer_work(spec, train), dom,
                                peaks, steps, clocks=clk(win), rec=rec, **kw)
        torch.cuda.empty_cache()

    entry("c1_fp32_fwd", "1D causal layer fwd, fp32, L=4096 d=256 4x64 P=64", S.spec_c1(), 0,
          False, 20, ffma=ffma)
    entry("c2_layer_fwd_bwd", "1D causal layer fwd+bwd, bf16, L=65536 d=1024 16x64 P=64",
          S.spec_c2(), 1, True, 10)
    entry("lm_history_fwd_bwd", "1D causal layer fwd+bwd with 64-wide tokens and 512-wide "
          "proxies (the language model's history stream), bf16, L=1048576 8x64 heads P=64",
          S.spec_lm_history(), 6, True, 10)
    for key, kw in (("mlp_interaction_fwd_bwd", dict(interact=S.F_MLP)),
                    ("rope_attention_fwd_bwd", dict(rope=1))):
        sv = S.LayerSpec(batch=1, L=262144, d=1024, n_heads=16, P=64, levels=2, k1=8, k2=8, **kw)
        what = ("single-proxy MLP interaction (hidden 4d, SiLU)" if "mlp" in key
                else "proxy attention with RoPE on queries and keys")
        entry(key, f"1D causal layer fwd+bwd with {what}, bf16, L=262144 d=1024 16x64 P=64 8x8",
              sv, 7, True, 10)
    out["segments_fwd_bwd"] = measure_segments(torch, pf, S, peaks, warmup, clk)
    torch.cuda.empty_cache()
    entry("cross_layer_fwd_bwd", "1D causal layer fwd+bwd with gated cross-attention injection "
          "(Eq. inj-cross), bf16, L=262144 d=1024 16x64 P=64 8x8", S.spec_cross_layer(), 5,
          True, 5)
    entry("c5_2d_fwd_bwd", "2D bidirectional layer fwd+bwd, bf16, B=4 512x512 d=512 8x64 8x8 "
          "patches", S.spec_c5(), 4, True, 5)
    specs, params = [], []
    for i, P in enumerate(S.C3_RATIOS):
        k1, k2 = S.default_factors(P)
        sp = S.LayerSpec(batch=1, L=262144, d=1024, n_heads=16, P=P, levels=2, k1=k1, k2=k2)
        specs.append(sp)
        params.append(S.make_layer_params(sp, 2 + 10 * i))
    st = ProxyStack(specs, params)
    inp = S.make_layer_inputs(specs[0], 2, with_grads=True)
    X = to_device(inp["X"], torch.bfloat16)
    G = to_device(inp["G"], torch.bfloat16)
    del inp

    def stack_step():
        st.forward(X)
        st.backward(G)
    ms, rec, dom, win = timed_steps(torch, pf, stack_step, 3, warmup)
    work = [sum(w) for w in zip(*(layer_work(sp) for sp in specs))]
    out["c3_stack_fwd_bwd"] = config_entry(
        "12-layer causal stack fwd+bwd, bf16, L=262144 d=1024 16x64, P=16..256 two-level",
        specs[0].L, ms, work, dom, peaks, 3, clocks=clk(win), rec=rec)
    del G
    out["prefill"] = measure_prefill(torch, pf, S, peaks, warmup, specs, params, st, X, clk)
    del st, X, params
    torch.cuda.empty_cache()
    return out


SEGMENTS = [(131072, 256, 16, 16), (98304, 64, 8, 8), (32768, 16, 4, 4)]


def measure_segments(torch, pf, S, peaks, warmup, clk):
    """Temporal-distance ratios (Sec. 3.6) on the 262144-token causal layer,
    d = 1024, 16x64 heads, two levels: the distant 131072 tokens in P = 256
    blocks, the next 98304 in P = 64, the recent 32768 in P = 16 (4096
    proxies, as many as uniform P = 64)."""
    from paper_2608_23463_gb300.segments import ProxySegmentLayer
    segs = SEGMENTS
    try:
        spec = S.LayerSpec(batch=1, L=262144, d=1024, n_heads=16, P=256, levels=2, k1=16, k2=16)
        shared, seg_prm = S.make_segment_params(1024, 16, 2, segs, 90)
        lay = ProxySegmentLayer(spec, segs, shared, seg_prm)
        g = torch.Generator(device="cuda").manual_seed(91)
        X = torch.randn(1, spec.L, 1024, device="cuda", generator=g).to(torch.bfloat16)
        G = torch.randn(1, spec.L, 1024, device="cuda", generator=g).to(torch.bfloat16)
        Xo, dX = torch.empty_like(X), torch.empty_like(X)

        def step():
            lay.forward(X, Xo)
            lay.backward(X, G, dX)
        ms, rec, dom, win = timed_steps(torch, pf, step, 5, warmup)
        return config_entry("1D causal layer fwd+bwd with temporal-distance ratios (P = 256 / 64 / "
                            "16 from distant to recent), bf16, L=262144 d=1024 16x64 two-level",
                            spec.L, ms, segments_work(1024, 16, 2, segs), dom, peaks, 5,
                            clocks=clk(win), rec=rec)
    except Exception as e:  # reported in the JSON line rather than ending the run
        return {"error": str(e).splitlines()[0][:200]}


def measure_prefill(torch, pf, S, peaks, warmup, specs, params, st, X, clk):
    """Prefill of the 12-layer causal stack over a 262144-token history
    (Sec. 3.8): the inference forward plus every layer's bulk proxy-cache
    fill, against a standard softmax-attention prefill of the same depth,
    width and history (per layer: the QKV projection, causal attention over
    all L tokens, the output projection).  The standard arm runs PyTorch's
    fused attention and cuBLAS, one layer timed and scaled by the depth; its
    FLOP floor at the measured (burst) bf16 peak is reported beside it."""
    from paper_2608_23463_gb300.decode import ProxyKVCache
    caches = []
    for i, s in enumerate(specs):
        ds = S.decode_spec_for_layer(s, s.L // s.P)
        dp = S.decode_params_for_layer(s, params[i], 200 + i)
        caches.append(ProxyKVCache(ds, dp, S.make_decode_state(ds, 0, [0], [0])))
    ms, rec, dom, win = timed_steps(torch, pf, lambda: st.prefill(X, caches), 3, warmup)
    L, d, n = specs[0].L, specs[0].d, len(specs)
    # the inference forward of every layer plus its cache rows (K and V, bf16)
    work = [sum(w) for w in zip(*(layer_work(sp, False) for sp in specs))]
    work[1] += sum(2 * (sp.L // sp.P) * sp.d * 2 for sp in specs)
    res = config_entry("causal stack prefill latency, 12 layers, L=262144 d=1024 16x64, "
                       "P=16..256 two-level, proxy caches filled", L, ms, work, dom, peaks, 3,
                       clocks=clk(win), rec=rec)
    res["latency_ms"] = ms
    del caches
    torch.cuda.empty_cache()
    # standard prefill, one layer
    std_flops = n * (2 * L * d * 4 * d + 2 * L * L * d)  # projections + causal QK^T and PV
    floor_ms = std_flops / (peaks["bf16_tflops"] * 1e12) * 1e3
    std = {"flops": std_flops, "floor_ms_at_measured_peak": floor_ms,
           "impl": "torch scaled_dot_product_attention (fused kernels only) + cuBLAS"}
    try:
        from torch.nn.attention import SDPBackend, sdpa_kernel
        g = torch.Generator(device="cuda").manual_seed(7)
        Xs = X.reshape(L, d)
        Wqkv = (torch.randn(3 * d, d, device="cuda", generator=g) / d ** 0.5).to(torch.bfloat16)
        Wo = (torch.randn(d, d, device="cuda", generator=g) / d ** 0.5).to(torch.bfloat16)
        nh = specs[0].n_heads

        def layer():
            qkv = Xs @ Wqkv.T
            q, k, v = (qkv[:, i * d:(i + 1) * d].reshape(1, L, nh, d // nh).transpose(1, 2)
                       for i in range(3))
            o = torch.nn.functional.scaled_dot_product_attention(q, k, v, is_causal=True)
            return o.transpose(1, 2).reshape(L, d) @ Wo.T

        backends = [SDPBackend.CUDNN_ATTENTION, SDPBackend.FLASH_ATTENTION,
                    SDPBackend.EFFICIENT_ATTENTION]
        with sdpa_kernel(backends):
            stream = torch.cuda.current_stream()
            layer()
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            for _ in range(2):
                layer()
            e1.record(stream)
            torch.cuda.synchronize()
        std["measured_ms"] = e0.elapsed_time(e1) / 2 * n
        res["speedup_vs_standard_measured"] = std["measured_ms"] / ms
    except Exception as e:  # the fused attention may be missing for this GPU
        std["measured_ms"] = None
        std["unavailable"] = str(e).splitlines()[0][:200]
    res["standard_attention_prefill"] = std
    res["speedup_vs_standard_floor"] = floor_ms / ms
    return res




def run_case(args):
    """A small run of one workload's step for profiler captures: W warm-up
    steps, then K steps; prints the mean step time."""
    import dataclasses

    import torch

    import paper_2608_23463_gb300 as pf
    import pf_synth as S
    from paper_2608_23463_gb300.layer import ProxyLayer, to_device
    pf.build()
    stream = torch.cuda.current_stream()
    if args.case == "decode":
        spec, ms, _, _, _, _ = measure_decode(torch, pf, S, max(args.steps, 1))
        print(json.dumps({"case": "decode", "ms_per_step": ms}), flush=True)
        return
    spec = {"layer": S.spec_c3_layer(64), "c1": S.spec_c1(), "c2": S.spec_c2(), "c5": S.spec_c5(),
            "cross": S.spec_cross_layer(), "lm_history": S.spec_lm_history()}[args.case]
    if args.batch:
        spec = dataclasses.replace(spec, batch=args.batch)
    if args.L:
        spec = dataclasses.replace(spec, L=args.L)
    train = spec.dtype == S.BF16  # the fp32 layer is forward-only
    dt = torch.bfloat16 if train else torch.float32
    inp = S.make_layer_inputs(spec, 2)
    lay = ProxyLayer(spec, inp)
    X = to_device(inp["X"], dt)
    G = to_device(inp["G"], dt)
    t = to_device(inp["t"], torch.float32) if "t" in inp else None
    del inp
    Xo, dX = lay.empty_act(), lay.empty_act()

    def step():
        lay.forward(X, None, t, X_out=Xo, train=train)
        if train:
            lay.backward(X, G, None, t, dX=dX)
    for _ in range(max(args.warmup, 1)):
        step()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        step()
    e1.record(stream)
    torch.cuda.synchronize()
    pf.pf_sync_check(stream.cuda_stream)
    ms = e0.elapsed_time(e1) / max(args.steps, 1)
    pf.pf_timing_enable(True)  # per-kernel breakdown of one more step
    step()
    torch.cuda.synchronize()
    t = pf.pf_timing_collect()
    pf.pf_timing_enable(False)
    pf.pf_sync_check(stream.cuda_stream)
    top = sorted(t.items(), key=lambda kv: -kv[1]["ms"])[:24]
    print(json.dumps({"case": args.case, "batch": spec.batch, "L": spec.L, "ms_per_step": ms,
                      "kernels_ms": {k: round(v["ms"], 4) for k, v in top}}), flush=True)


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            return json.load(f), "measured"
    return PEAKS_FALLBACK, "fallback"


def run_ours(args, rank: int, world: int, local_rank: int):
    import numpy as np
    import torch
    import torch.distributed as dist

    import paper_2608_23463_gb300 as pf
    import pf_synth as S
    from paper_2608_23463_gb300.layer import ProxyLayer, to_device

    torch.cuda.set_device(local_rank)
    pf.build()
    spec = workload_spec(args.L)
    inp = S.make_layer_inputs(spec, rank_seed(rank))
    lay = ProxyLayer(spec, inp)
    X = to_device(inp["X"], torch.bfloat16)
    G = to_device(inp["G"], torch.bfloat16)
    del inp
    Xo, dX = lay.empty_act(), lay.empty_act()
    stream = torch.cuda.current_stream()

    def step():
        lay.forward(X, X_out=Xo)
        lay.backward(X, G, dX=dX)

    for _ in range(max(args.warmup, 3)):
        step()
    pf.pf_sync_check(stream.cuda_stream)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()

    sampler = ClockSampler(gpu_smi_id(torch, local_rank)) if rank == 0 else None
    time.sleep(0.3)
    # the timed steps run with per-launch timing off (no extra events in the
    # stream); the per-kernel breakdown comes from a separate pass below
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    if sampler:
        sampler.mark(True)
    e0.record(stream)
    for _ in range(args.steps):
        step()
    e1.record(stream)
    torch.cuda.synchronize()
    if sampler:
        sampler.mark(False)
    if world > 1:
        dist.barrier()
    ms = e0.elapsed_time(e1) / args.steps
    pf.pf_sync_check(stream.cuda_stream)
    clocks = sampler.window(sampler.t0, sampler.t1) if sampler else None
    # breakdown pass: the same steps with CUDA events around every launch,
    # scaled to the timed step count
    bsteps = min(args.steps, 10)
    pf.pf_timing_enable(True)
    for _ in range(bsteps):
        step()
    torch.cuda.synchronize()
    timing = pf.pf_timing_collect()
    pf.pf_timing_enable(False)
    pf.pf_sync_check(stream.cuda_stream)
    for v in timing.values():
        v["ms"] *= args.steps / bsteps
        v["launches"] = v["launches"] * args.steps // bsteps
    ms = max_over_ranks(ms, world)
    tokens_per_step = spec.batch * spec.L * world
    value = job_throughput(spec.batch * spec.L, world, ms)
    launches = sum(v["launches"] for v in timing.values())

    # ---- end to end: pinned host inputs in, results out, every step.  The
    # copies run on their own streams with double-buffered device tensors, so
    # step i's device-to-host read and step i+1's host-to-device copy overlap
    # the layer's kernels (as a training loop that prefetches its next batch).
    Xh = X.cpu().pin_memory()
    Gh = G.cpu().pin_memory()
    Xoh = torch.empty_like(Xh).pin_memory()
    dXh = torch.empty_like(Xh).pin_memory()
    Xd = [torch.empty_like(X) for _ in range(2)]
    Gd = [torch.empty_like(G) for _ in range(2)]
    Xod = [torch.empty_like(Xo) for _ in range(2)]
    dXd = [torch.empty_like(dX) for _ in range(2)]
    h2d, d2h = torch.cuda.Stream(), torch.cuda.Stream()
    ev_in = [torch.cuda.Event() for _ in range(2)]    # inputs of buffer k on the device
    ev_done = [torch.cuda.Event() for _ in range(2)]  # the layer is done with buffer k
    ev_out = [torch.cuda.Event() for _ in range(2)]   # outputs of buffer k read back

    def e2e_step(i):
        k = i & 1
        with torch.cuda.stream(h2d):
            h2d.wait_event(ev_done[k])  # step i-2 no longer reads input buffer k
            Xd[k].copy_(Xh, non_blocking=True)
            Gd[k].copy_(Gh, non_blocking=True)
            ev_in[k].record(h2d)
        stream.wait_event(ev_in[k])
        stream.wait_event(ev_out[k])  # step i-2's outputs have been read back
        lay.forward(Xd[k], X_out=Xod[k])
        lay.backward(Xd[k], Gd[k], dX=dXd[k])
        ev_done[k].record(stream)
        with torch.cuda.stream(d2h):
            d2h.wait_event(ev_done[k])
            Xoh.copy_(Xod[k], non_blocking=True)
            dXh.copy_(dXd[k], non_blocking=True)
            ev_out[k].record(d2h)

    for i in range(2):
        e2e_step(i)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    e0.record(stream)
    h2d.wait_event(e0)
    for i in range(args.e2e_steps):
        e2e_step(i)
    stream.wait_event(ev_out[(args.e2e_steps - 1) & 1])
    e1.record(stream)
    torch.cuda.synchronize()
    ms_e2e = e0.elapsed_time(e1) / args.e2e_steps
    ms_e2e = max_over_ranks(ms_e2e, world)
    pf.pf_sync_check(stream.cuda_stream)
    act_bytes = spec.batch * spec.L * spec.d * 2
    del Xh, Gh, Xoh, dXh, Xd, Gd, Xod, dXd
    decode_result = None
    if not args.no_decode:
        del lay, X, G, Xo, dX
        torch.cuda.empty_cache()
        decode_result = measure_decode(torch, pf, S, args.decode_steps)
    configs_result = None
    ffma = measure_ffma_peak(torch, pf) if not args.no_configs else None
    if not args.no_configs:
        if not args.no_decode:
            torch.cuda.empty_cache()
        else:
            del lay, X, G, Xo, dX
            torch.cuda.empty_cache()
        configs_result = measure_configs(torch, pf, S, load_peaks()[0], max(args.warmup, 3),
                                         sampler, ffma)
    if sampler:
        sampler.stop()
    if rank != 0:
        return

    peaks, peak_src = load_peaks()
    comp_peak, comp_src = compute_peak(peaks, clocks)
    # dominant kernel: largest share of the timed region
    dom, dv = max(timing.items(), key=lambda kv: kv[1]["ms"])
    avg_s = dv["ms"] / dv["launches"] / 1e3
    units = spec.batch * spec.L
    if dv["flops"] > 0 and not dom.startswith(("inj_bwd", "colsum", "copy", "pad")):
        achieved = dv["flops"] / avg_s / 1e12
        roof = {"bound": "tensor", "achieved": achieved, "peak": comp_peak, "unit": "TFLOP/s",
                "frac": achieved / comp_peak, "traffic": traffic_from_profile(dom, units),
                "kernel": dom, "launches": dv["launches"], "avg_us": avg_s * 1e6,
                "flops_per_launch": dv["flops"],
                "peak_source": f"{peak_src} {comp_src} (of measured)"}
    else:
        achieved = dv["bytes"] / avg_s / 1e9
        peak = peaks["hbm_gbs"]
        roof = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                "frac": achieved / peak, "traffic": traffic_from_profile(dom, units),
                "kernel": dom, "launches": dv["launches"], "avg_us": avg_s * 1e6,
                "bytes_per_launch": dv["bytes"], "peak_source": f"{peak_src} hbm_gbs"}
    step_flops, step_bytes = layer_work(spec)
    t_c = step_flops / (comp_peak * 1e12) * 1e3
    t_b = step_bytes / (peaks["hbm_gbs"] * 1e9) * 1e3
    roof_ms = max(t_c, t_b)
    total_ms = sum(v["ms"] for v in timing.values())
    breakdown = {k: {"ms_per_step": v["ms"] / args.steps, "share": v["ms"] / total_ms,
                     "launches_per_step": v["launches"] / args.steps}
                 for k, v in sorted(timing.items(), key=lambda kv: -kv[1]["ms"])}
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
            "data": "synthetic", "config": config_dict(spec),
            "roofline": roof,
            "layer_roofline": {"flops_per_step": step_flops, "bytes_per_step": step_bytes,
                               "bound": "tensor" if t_c >= t_b else "hbm",
                               "roofline_ms": roof_ms, "frac": roof_ms / ms,
                               "peaks": f"{peak_src}: bf16 {comp_peak:.1f} TFLOP/s "
                                        f"({comp_src}), HBM {peaks['hbm_gbs']} GB/s",
                               "work": "algorithmic (Eq. complexity, Sec. 4)"},
            "e2e": {"value": tokens_per_step / (ms_e2e / 1e3), "unit": UNIT,
                    "h2d_bytes_per_step": 2 * act_bytes, "d2h_bytes_per_step": 2 * act_bytes,
                    "ms_per_step": ms_e2e,
                    "copies": "pinned host X, dX_out in and X_out, dX out every step, on two "
                              "copy streams overlapping the previous / next step's kernels"},
            "gpu_launches": launches, "clocks": clocks,
            "kernels": {k: round(v["ms_per_step"], 4) for k, v in list(breakdown.items())[:6]}}
    detail = {"kernels": breakdown}
    if not args.no_decode:
        dspec, dms, dms_direct, app_ms, dbytes, dkern = decode_result
        dec = {
            "metric": "proxy-KV decode new tokens/s per layer (B=8, 16384 cached proxies, "
                      "d=2048, 16x128 heads, open block 0..63)",
            "value": dspec.batch / (dms / 1e3), "unit": "tokens/s", "ms_per_step": dms,
            "steps": args.decode_steps,
            "roofline": {"bound": "hbm", "achieved": dbytes / (dms / 1e3) / 1e9,
                         "peak": peaks["hbm_gbs"], "unit": "GB/s",
                         "frac": dbytes / (dms / 1e3) / 1e9 / peaks["hbm_gbs"],
                         "bytes_per_step": dbytes},
            "timing": "CUDA graph of one step, replayed back to back; events per 64-step span",
            "direct_call_ms_per_step": dms_direct,
            "append_ms": app_ms, "kernels_ms_per_step": dkern}
        detail["decode"] = dec
        line["decode"] = {"tok_s": round(dec["value"]), "ms": round(dms, 4),
                          "frac_hbm": round(dec["roofline"]["frac"], 3),
                          "direct_ms": round(dms_direct, 4), "append_ms": round(app_ms, 4)}
    if configs_result is not None:
        detail["configs"] = configs_result
        detail["ffma_tflops_measured"] = ffma
        compact = {}
        for k, v in configs_result.items():
            if "roofline" not in v:
                compact[k] = v
                continue
            r = v["roofline"]
            compact[k] = {"tok_s": float(f"{v['value']:.4g}"), "ms": round(v["ms_per_step"], 4),
                          "frac": round(r["frac"], 3), "bound": r["bound"],
                          "top": r.get("kernel")}
        compact["ffma_tflops"] = round(ffma, 1) if ffma else None
        line["configs"] = compact
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline_subprocess()
    if args.detail:
        with open(args.detail, "w") as f:
            json.dump(detail, f, indent=1)
    print(json.dumps(line), flush=True)


def main():
    args = parse_args()
    rank = int(os.environ.get("RANK", 0))
    world = int(os.environ.get("WORLD_SIZE", 1))
    local_rank = int(os.environ.get("LOCAL_RANK", 0))
    sys.path.insert(0, ROOT)
    if args.impl == "reference":
        run_reference(args, rank)
        return
    if args.case:
        run_case(args)
        return
    import torch.distributed as dist
    if world > 1:
        import torch
        torch.cuda.set_device(local_rank)
        dist.init_process_group("nccl")
    try:
        run_ours(args, rank, world, local_rank)
    finally:
        if world > 1:
            dist.destroy_process_group()


if __name__ == "__main__":
    main()
