"""Benchmark of the StateKV per-frame video-prefill step on GB300.

A step is one frame of the workload: every layer (and stream) runs the whole
hot path -- frame attention with fused importance, top-B state selection and
gather, decode-cache append -- through ``statekv_prefill_frame``.  Before the
timed steps the state is filled (the frames whose pool still fits in B run
untimed), so the timed frames are the steady state: "given the preceding
cache, process one more frame" (App. B's protocol).

Prints one JSON line.  ``--impl reference`` times the CPU oracle instead (the
paper ships no implementation; the oracle is the reference arm).
"""
from __future__ import annotations

import argparse
import dataclasses
import hashlib
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

DEFAULT_WORKLOAD = "qwen7b_stack"
METRIC = "frames/s and p50 per-frame \u00b5s at 7B shape; % of BF16 tensor peak"
WORKLOAD_TEXT = {
    "qwen7b_stack": "28-layer Qwen2-7B-shaped stack: 28 q / 4 kv heads, head_dim 128, bf16, "
                    "196 tokens/frame, state capacity 2048, 256-frame video",
    "qwen7b_layer": "one Qwen2-7B-shaped attention layer: 28 q / 4 kv heads, head_dim 128, bf16, "
                    "196 tokens/frame, state capacity 1568, 64-frame video",
    "qwen72b_stack": "80-layer 72B-shaped stack: 64 q / 8 kv heads, head_dim 128, bf16, "
                     "196 tokens/frame, state capacity 4096, 512-frame video",
    "qwen7b_8streams": "8 concurrent 7B-shaped streams x 28 layers, 28 q / 4 kv heads, head_dim 128, "
                       "bf16, 196 tokens/frame, state capacity 2048, 1024 frames each",
    "toy": "toy layer: 4 q / 1 kv heads, head_dim 64, 16 tokens/frame, state capacity 32",
}
KERNEL_SOURCE = os.path.join(ROOT, "paper_2605_31598_gb300", "csrc", "attn_kernel.cu")
# DRAM bytes (dram__bytes_read.sum + dram__bytes_write.sum) of one attention
# launch, from one ncu capture per workload, keyed by the workload and the
# first 16 hex digits of the sha256 of the attention-kernel source it was taken
# on.  A workload or kernel source with no capture reports null.
K1_DRAM_BYTES = {
    ("qwen7b_stack", "c286b2182a710e41"): 197721088,
    ("qwen72b_stack", "c286b2182a710e41"): 2047845120,
    ("qwen7b_8streams", "c286b2182a710e41"): 1727971328,
}


FLATNESS_MIN_FRAMES = 64
KERNEL_PASS_STEPS = 64  # steps of the profiled pass that times each kernel
# --curve generates inputs in chunks of at most this many bytes
CURVE_CHUNK_BYTES = 24e9


def log(*a):
    print(*a, file=sys.stderr, flush=True)


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return p["hbm_gbs"], p["bf16_tflops"], p.get("bf16_tflops_sustained"), "measured"
    return 6800.0, 1900.0, 1700.0, "fallback"


def attn_flops(shape, count):
    """Algorithmic FLOPs of the frame attention for one (stream, layer):
    QK^T and PV over the visible pairs, 4 d Hq (T count + T (T + 1) / 2).
    The QK^T recompute of the two-pass design is not counted."""
    T, d, Hq = shape.tokens_per_frame, shape.head_dim, shape.num_q_heads
    return 4.0 * d * Hq * (T * count + T * (T + 1) / 2)


def kernel_source_hash():
    with open(KERNEL_SOURCE, "rb") as f:
        return hashlib.sha256(f.read()).hexdigest()[:16]


def recorded_traffic(workload):
    """DRAM bytes per attention launch captured for this workload on the
    current kernel source, or None."""
    return K1_DRAM_BYTES.get((workload, kernel_source_hash()))


class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled in the background."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_id: str):
        self.samples = []
        self.proc = None
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", gpu_id, f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "50"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except (OSError, FileNotFoundError):
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.samples.append((time.time(), [x.strip() for x in line.split(",")]))

    def stop(self):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self, t0, t1, pad=0.3):
        if not self.samples:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no nvidia-smi samples"],
                    "samples": 0}
        win = [s for (t, s) in self.samples if t0 - pad <= t <= t1 + pad]
        if not win:  # timed region shorter than the sampling period: nearest samples
            mid = 0.5 * (t0 + t1)
            win = [min(self.samples, key=lambda x: abs(x[0] - mid))[1]]
        sm = [float(s[0]) for s in win if s[0].replace(".", "").isdigit()]
        mx = [float(s[1]) for s in win if s[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for s in win for i in range(4)
                          if len(s) > 4 + i and s[4 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(win),
                "power_w_max": max((float(s[2]) for s in win
                                    if s[2].replace(".", "").isdigit()), default=None)}


def gpu_sampler(device):
    """A clock sampler on the GPU behind ``device`` (by UUID when torch knows it)."""
    import torch

    props = torch.cuda.get_device_properties(device)
    gpu_id = f"GPU-{props.uuid}" if getattr(props, "uuid", None) else str(device.index or 0)
    return ClockSampler(gpu_id)


def dist_setup():
    import torch
    import torch.distributed as dist

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        backend = "nccl" if torch.cuda.is_available() else "gloo"
        if backend == "nccl":
            torch.cuda.set_device(local)
        dist.init_process_group(backend)
    return world, rank, local


def max_over_ranks(x: float, world: int, device) -> float:
    if world == 1:
        return x
    import torch
    import torch.distributed as dist

    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def barrier(world):
    if world > 1:
        import torch.distributed as dist

        dist.barrier()


# ---------------------------------------------------------------- oracle legs
def _oracle_units(shape, n_units, seed, g):
    """Prepared oracle calls of ``n_units`` (layer, KV head) units of one
    steady-state frame (state full with B entries), ``g`` query heads each."""
    import numpy as np
    import torch

    import oracle
    from paper_2605_31598_gb300.inputs import frame_qkv

    T, Hq, Hkv, d, B, L = (shape.tokens_per_frame, shape.num_q_heads, shape.num_kv_heads,
                           shape.head_dim, shape.state_capacity, shape.num_layers)
    G = Hq // Hkv
    n_frame = math.ceil(B / T) + 1 if B > 0 else 1
    calls = []
    for i in range(n_units):
        layer, h = (i // Hkv) % L, i % Hkv
        q, k, v = frame_qkv(shape, n_frame, layer=layer, seed=seed)
        qb = np.ascontiguousarray(oracle.as_bf16_bits(q)[:, h * G: h * G + g])
        kb = np.ascontiguousarray(oracle.as_bf16_bits(k)[:, h: h + 1])
        vb = np.ascontiguousarray(oracle.as_bf16_bits(v)[:, h: h + 1])
        lay = oracle.OracleLayer(g, 1, d, T, B, n_frame)
        gen = torch.Generator().manual_seed(seed + i)
        sk = oracle.as_bf16_bits((torch.randn((1, B, d), generator=gen) * d ** -0.5).bfloat16())
        sv = oracle.as_bf16_bits((torch.randn((1, B, d), generator=gen) * d ** -0.5).bfloat16())
        lay.set_state(np.array([B], np.int32), np.arange(B, dtype=np.int64)[None], sk, sv,
                      (n_frame - 1) * T)
        calls.append((lay, qb, kb, vb))
    return calls


def oracle_units_timing(shape, n_units, seed=0, q_heads=None, threads=1):
    """Times the CPU oracle on ``n_units`` (layer, KV head) units of one
    steady-state frame.  Each unit is the oracle called on one KV head's query
    group; ``q_heads`` < G restricts the group.  With ``threads`` > 1 the
    units run concurrently on that many host threads (the oracle's C loop runs
    without the Python lock) and the wall time is returned.  Returns
    (seconds, fraction of a whole frame step processed)."""
    Hq, Hkv, L = shape.num_q_heads, shape.num_kv_heads, shape.num_layers
    G = Hq // Hkv
    g = G if q_heads is None else q_heads
    calls = _oracle_units(shape, n_units, seed, g)
    frac = n_units * g / float(L * Hkv * G)
    if threads <= 1:
        total = 0.0
        for lay, qb, kb, vb in calls:
            t0 = time.perf_counter()
            lay.prefill_frame(qb, kb, vb)
            total += time.perf_counter() - t0
        return total, frac
    import concurrent.futures as cf

    with cf.ThreadPoolExecutor(max_workers=threads) as ex:
        t0 = time.perf_counter()
        list(ex.map(lambda c: c[0].prefill_frame(*c[1:]), calls))
        return time.perf_counter() - t0, frac


def run_reference(args, world, rank):
    """The reference arm: the CPU oracle, timed on the host cores."""
    if rank != 0:
        return
    import oracle
    from paper_2605_31598_gb300.inputs import WORKLOADS

    oracle.build()
    shape = WORKLOADS[args.workload]
    G = shape.num_q_heads // shape.num_kv_heads
    cores = os.cpu_count() or 1
    # size each step so the whole run stays within about two minutes: one
    # unit per host thread, each with g of the G query heads
    t_one, _ = oracle_units_timing(shape, 1, q_heads=1)
    budget = 120.0 / max(1, args.steps + args.warmup)
    g = max(1, min(G, int(budget / max(t_one, 1e-6))))
    for _ in range(args.warmup):
        oracle_units_timing(shape, cores, q_heads=g, threads=cores)
    secs, frac = 0.0, 0.0
    for _ in range(args.steps):
        s, f = oracle_units_timing(shape, cores, q_heads=g, threads=cores)
        secs += s
        frac += f
    value = shape.num_streams * frac / secs
    sample = (f"each step: the oracle on {cores} (layer, KV head) units of a steady-state frame "
              f"(state full, B={shape.state_capacity}), {g} of the {G} query heads each, one "
              f"unit per host thread; frames/s = fraction of a frame processed / wall time")
    line = {
        "impl": "reference", "metric": METRIC,
        "value": value, "unit": "frames/s", "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * secs / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": {"workload": WORKLOAD_TEXT[args.workload]},
        "cpu_baseline": {"value": value, "unit": "frames/s", "cores": cores, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": value, "unit": "frames/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------- our arm
def run_ours(args, world, rank, local):
    import torch

    from paper_2605_31598_gb300 import StateKV, make_config
    from paper_2605_31598_gb300.inputs import WORKLOADS, batch_qkv

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (no CPU fallback exists)")
    device = torch.device("cuda", local)
    torch.cuda.set_device(device)
    base = WORKLOADS[args.workload]
    T, B = base.tokens_per_frame, base.state_capacity
    S, L, Hkv = base.num_streams, base.num_layers, base.num_kv_heads
    fill = math.ceil(B / T) if B > 0 else 0  # frames until the state holds B tokens
    nframes = fill + args.warmup + args.steps
    # the kernel-timing pass after the timed steps replays their inputs
    kpass = min(args.steps, KERNEL_PASS_STEPS)
    max_frames = args.max_frames or base.max_frames
    if max_frames < nframes + kpass:
        max_frames = nframes + kpass
    shape = dataclasses.replace(base, max_frames=max_frames)
    seed = args.seed + 1000 * rank
    log(f"[bench] rank {rank}: generating {nframes} frames of {args.workload} inputs")
    frames = [batch_qkv(shape, n, streams=range(S), layers=range(L), seed=seed, device=device)
              for n in range(1, nframes + 1)]
    sel = SELECTIONS[args.selection]
    eng = StateKV(make_config(shape, selection=sel))
    out = torch.empty_like(frames[0][0])
    imp = (torch.empty((S, L, Hkv, B + T), dtype=torch.float32, device=device)
           if sel != 1 else None)

    def step(n):
        q, k, v = frames[n]
        rc = eng.prefill_frame(q, k, v, out, imp)
        if rc != 0:
            raise RuntimeError(f"statekv_prefill_frame returned {rc} "
                               f"(device word 0x{eng.device_error():x}) at frame {n + 1}")

    eng.profile(True)  # creates the event pool outside the timed region
    eng.profile(False)
    for n in range(fill + args.warmup):
        step(n)
    torch.cuda.synchronize()

    sampler = gpu_sampler(device)
    time.sleep(0.3)
    st = torch.cuda.current_stream()
    # one event per step boundary: step i runs between bounds[i] and bounds[i + 1]
    bounds = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps + 1)]
    barrier(world)
    torch.cuda.synchronize()
    t_wall0 = time.time()
    bounds[0].record(st)
    for i in range(args.steps):
        step(fill + args.warmup + i)
        bounds[i + 1].record(st)
    torch.cuda.synchronize()
    t_wall1 = time.time()
    barrier(world)
    # Kernel durations come from a second pass over the same inputs with the
    # library's per-launch events on: those events sit between the kernels and
    # would lengthen the timed steps above, so they are kept out of them.
    eng.profile(True)
    for i in range(kpass):
        step(fill + args.warmup + i)
    torch.cuda.synchronize()
    t_wall2 = time.time()
    prof = eng.profile_read()
    eng.profile(False)
    time.sleep(0.3)
    sampler.stop()
    per_step = [bounds[i].elapsed_time(bounds[i + 1]) for i in range(args.steps)]
    total_ms = bounds[0].elapsed_time(bounds[-1])
    total_ms_max = max_over_ranks(total_ms, world, device)
    assert eng.sync() == 0

    hbm, tf_burst, tf_sust, peak_kind = peaks()
    # dominant kernel: frame attention + importance (kind 1)
    k1_launches, k1_ms = prof[1]
    k1_avg_s = k1_ms / max(k1_launches, 1) * 1e-3
    flops = S * L * attn_flops(shape, B)
    achieved = flops / k1_avg_s / 1e12
    traffic = recorded_traffic(args.workload)
    a_launches, a_ms = prof[0]
    s_launches, s_ms = prof[2]
    d = shape.head_dim
    append_bytes = 2 * 2 * S * L * Hkv * T * d * 2  # read + write K and V rows
    # The append shares the selection's launch (with the recency window it is a
    # launch of its own on a side stream, off the critical path); the shares are
    # of the two kernels in series.
    kernels = {
        "frame_attn_lse_importance": {"avg_us": 1e6 * k1_avg_s, "tflops": achieved,
                                      "share": k1_ms / max(1e-9, k1_ms + s_ms)},
        "decode_cache_append": {"bytes": append_bytes, "launched_with": "state_select_gather"},
        "state_select_gather": {"avg_us": 1e3 * s_ms / max(s_launches, 1),
                                "share": s_ms / max(1e-9, k1_ms + s_ms)},
    }
    if a_launches:
        kernels["decode_cache_append"] = {"span_us": 1e3 * a_ms / a_launches, "bytes": append_bytes,
                                          "concurrent_with": "frame_attn_lse_importance (side stream)"}
    value = world * S * args.steps / (total_ms_max * 1e-3)
    ps = sorted(per_step)
    # flat per-frame cost: slope of a linear fit of per-frame time against the
    # frame index, and the p50 of the first 32 timed frames vs the last half
    first = fill + args.warmup + 1
    idx = list(range(first, first + args.steps))
    n = len(per_step)
    mx, my = sum(idx) / n, sum(per_step) / n
    var = sum((x - mx) ** 2 for x in idx)
    slope = sum((x - mx) * (y - my) for x, y in zip(idx, per_step)) / var if var > 0 else 0.0
    early = sorted(per_step[:32])
    late = sorted(per_step[n // 2:])
    # a per-100-frame slope needs a window of comparable length to mean anything
    flatness = {"frames": f"{first}..{first + n - 1}",
                "slope_pct_per_100_frames": (100.0 * 100.0 * slope / my
                                             if my > 0 and n >= FLATNESS_MIN_FRAMES else None),
                "p50_first32_us": 1e3 * early[len(early) // 2],
                "p50_last_half_us": 1e3 * late[len(late) // 2]}
    if n < FLATNESS_MIN_FRAMES:
        flatness["note"] = (f"slope omitted: {n} timed frames (< {FLATNESS_MIN_FRAMES}); "
                            "bench.py --curve measures the per-frame cost over whole videos")
    line = {
        "metric": METRIC,
        "value": value,
        "unit": "frames/s",
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": total_ms_max / args.steps,
        "p50_us_per_frame": 1e3 * ps[len(ps) // 2],
        "p90_us_per_frame": 1e3 * ps[min(len(ps) - 1, int(0.9 * len(ps)))],
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "bf16",
        "data": "synthetic",
        "config": {"workload": WORKLOAD_TEXT[args.workload], "streams": S, "layers": L,
                   "selection": SELECTION_TEXT[sel],
                   "steady_state_frames": f"{fill + args.warmup + 1}..{nframes}",
                   "l2": "no flush: each step reads fresh Q/K/V and the full state "
                         f"(~{(2 * S * L * Hkv * B * d * 2 + S * L * T * (shape.num_q_heads + 2 * Hkv) * d * 2) / 1e6:.0f} MB "
                         "per step) > 129 MB L2",
                   "parallelism": f"replicas{world}" if world > 1 else "single"},
        "roofline": {"bound": "tensor", "achieved": achieved,
                     "peak": tf_burst, "unit": "TFLOP/s", "frac": achieved / tf_burst,
                     "peak_kind": f"{peak_kind} bf16 dense burst",
                     "frac_of_sustained": (achieved / tf_sust) if tf_sust else None,
                     "traffic": traffic,
                     "kernel": "frame_attn_lse_importance",
                     "flops_per_launch": flops},
        "kernels": kernels,
        "flatness": flatness,
        "gpu_launches": (4 if a_launches else 2) * args.steps,
    }
    line["config"]["kernel_timing"] = (f"kernel durations from a second pass of {kpass} steps over the same "
                                       "inputs with per-launch CUDA events on the launching streams; the "
                                       "timed steps carry one event per step boundary")
    clocks = sampler.summary(t_wall0, t_wall1)
    clocks["kernel_pass"] = sampler.summary(t_wall1, t_wall2)
    line["clocks"] = clocks

    # end to end through the host-buffer entry point (copies inside the timed region)
    if not args.no_e2e:
        line["e2e"] = run_e2e(args, shape, fill, seed, device, frames)
    del frames
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        import oracle

        oracle.build()
        cores = os.cpu_count() or 1
        n_units = 2 * cores
        secs, frac = oracle_units_timing(shape, n_units, seed=seed, threads=cores)
        s1, f1 = oracle_units_timing(shape, 4, seed=seed)
        line["cpu_baseline"] = {
            "value": S * frac / secs, "unit": "frames/s", "cores": cores, "kind": "oracle",
            "sample": f"{n_units} (layer, KV head) units of one steady-state frame "
                      f"({frac:.3f} of a frame) on {cores} host threads, {secs:.1f} s wall, fp64; "
                      "scaled to frames/s",
            "single_thread": {"value": S * f1 / s1, "unit": "frames/s",
                              "sample": f"4 units ({f1:.3f} of a frame), {s1:.1f} s"}}
    if rank == 0:
        print(json.dumps(line), flush=True)


def run_e2e(args, shape, fill, seed, device, frames):
    """Same steps through statekv_prefill_frames_host, the streaming host-buffer
    call: every step copies that frame's Q/K/V from pinned host memory and its
    output (and importance) back, all inside the timed region; the copies of
    frame i + 1 and i - 1 overlap the step of frame i."""
    import torch

    from paper_2605_31598_gb300 import StateKV, make_config

    S, L, Hkv, T, B = (shape.num_streams, shape.num_layers, shape.num_kv_heads,
                       shape.tokens_per_frame, shape.state_capacity)
    steps = min(args.steps, 64)
    n_total = fill + args.warmup + steps
    host = [tuple(x.cpu().pin_memory() for x in frames[n]) for n in range(n_total)]
    # The first DMA from a freshly pinned page runs ~7x slower than later ones
    # (measured: 1.8 against 0.25 ms per frame's Q/K/V).  A streaming pipeline
    # reuses a warm ring of pinned staging buffers, so every buffer is copied
    # to the device once here, before the timed region.
    for n in range(n_total):
        for x, y in zip(frames[n], host[n]):
            x.copy_(y, non_blocking=True)
    torch.cuda.synchronize()
    sel = SELECTIONS[args.selection]
    # two output buffer sets, alternating by frame (the pipeline has two frames in flight)
    outs = [(torch.empty(host[0][0].shape, dtype=torch.bfloat16).pin_memory(),
             torch.empty((S, L, Hkv, B + T), dtype=torch.float32).pin_memory() if sel != 1 else None)
            for _ in range(2)]
    eng = StateKV(make_config(shape, host_staging=True, selection=sel))

    def run(first, count):
        frames_h = [host[n] + outs[n & 1] for n in range(first, first + count)]
        rc = eng.prefill_frames_host(frames_h)
        if rc != 0:
            raise RuntimeError(f"statekv_prefill_frames_host returned {rc}")

    run(0, fill + args.warmup)  # also DMA-touches both output sets
    torch.cuda.synchronize()
    st = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(st)
    run(fill + args.warmup, steps)
    e1.record(st)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    assert eng.sync() == 0
    h2d = sum(x.numel() * x.element_size() for x in host[0])
    d2h = outs[0][0].numel() * 2 + (outs[0][1].numel() * 4 if outs[0][1] is not None else 0)
    eng.close()
    return {"value": S * steps / (ms * 1e-3), "unit": "frames/s", "h2d_bytes_per_step": h2d,
            "d2h_bytes_per_step": d2h, "steps": steps,
            "api": "statekv_prefill_frames_host (pinned host buffers; copies in and out on "
                   "their own streams, overlapping the neighbouring frames' steps)",
            "staging": "one pinned input set per frame, each DMA-touched once before timing; "
                       "two output sets, alternating"}


def run_curve(args, local):
    """Per-frame cost against the frame index, StateKV next to exact full
    self-attention (Sec. 4.1's comparison, App. B's protocol: given the
    preceding cache, process one more frame).

    The frames' inputs are generated in chunks that fit in HBM, outside any
    timed region; the frames of a chunk then run back to back, each
    statekv_prefill_frame bracketed by CUDA events, so the GPU stays busy and
    the clocks sampled meanwhile are those of the timed work.  At sample
    frames statekv_full_attention_frame first runs on the same handle, over
    the decode cache that the earlier frames filled (twice; the second run is
    timed).  nvidia-smi clocks are sampled throughout; every 32-frame bin and
    every sample frame reports the median SM clock of the samples taken while
    it ran (the nearest sample when none fell inside).  Prints one JSON line.
    """
    import torch

    from paper_2605_31598_gb300 import StateKV, make_config
    from paper_2605_31598_gb300.inputs import WORKLOADS, batch_qkv

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (no CPU fallback exists)")
    device = torch.device("cuda", local)
    torch.cuda.set_device(device)
    shape = WORKLOADS[args.workload]
    if args.capacity is not None:  # the paper's wall-time sweep varies the state capacity
        shape = dataclasses.replace(shape, state_capacity=args.capacity)
    S, L, T, B = shape.num_streams, shape.num_layers, shape.tokens_per_frame, shape.state_capacity
    Hq, Hkv, d = shape.num_q_heads, shape.num_kv_heads, shape.head_dim
    N = args.frames or shape.max_frames
    shape = dataclasses.replace(shape, max_frames=max(N, shape.max_frames))
    samples = sorted({n for n in (1, 2, 4, 8, 16, 32, 64, 96, 128, 192, 256, 384, 512, 640, 768,
                                  896, 1024) if n <= N} | {N})
    frame_bytes = S * L * T * (Hq + 2 * Hkv) * d * 2
    chunk = max(1, min(N, int(CURVE_CHUNK_BYTES // frame_bytes)))
    eng = StateKV(make_config(shape))
    st = torch.cuda.current_stream()
    out = None
    step_ms, full_ms, wall = [0.0] * N, {}, [(0.0, 0.0)] * N
    full_wall = {}
    log(f"[curve] {args.workload}: {N} frames in chunks of {chunk}, full attention at {samples}")
    sampler = gpu_sampler(device)
    time.sleep(0.3)
    t_all0 = time.time()
    ev = lambda: torch.cuda.Event(enable_timing=True)
    for c0 in range(1, N + 1, chunk):
        c1 = min(N, c0 + chunk - 1)
        frames = [batch_qkv(shape, n, streams=range(S), layers=range(L), seed=args.seed,
                            device=device) for n in range(c0, c1 + 1)]
        if out is None:
            out = torch.empty_like(frames[0][0])
        torch.cuda.synchronize()
        base = ev()
        marks = []
        t0 = time.time()
        base.record(st)
        for n in range(c0, c1 + 1):
            q, k, v = frames[n - c0]
            fm = None
            if n in samples:
                for rep in range(2):  # second run timed: code and TMA descriptors warm
                    f0, f1 = ev(), ev()
                    f0.record(st)
                    rc = eng.full_attention_frame(q, k, v, out)
                    f1.record(st)
                    if rc != 0:
                        raise RuntimeError(f"statekv_full_attention_frame returned {rc} at frame {n}")
                fm = (f0, f1)
            e0, e1 = ev(), ev()
            e0.record(st)
            rc = eng.prefill_frame(q, k, v, out)
            e1.record(st)
            if rc != 0:
                raise RuntimeError(f"statekv_prefill_frame returned {rc} at frame {n}")
            marks.append((n, e0, e1, fm))
        torch.cuda.synchronize()
        for n, e0, e1, fm in marks:
            step_ms[n - 1] = e0.elapsed_time(e1)
            # wall-clock window of the frame: the chunk's start plus its GPU offset
            wall[n - 1] = (t0 + 1e-3 * base.elapsed_time(e0), t0 + 1e-3 * base.elapsed_time(e1))
            if fm is not None:
                full_ms[n] = fm[0].elapsed_time(fm[1])
                full_wall[n] = (t0 + 1e-3 * base.elapsed_time(fm[0]),
                                t0 + 1e-3 * base.elapsed_time(fm[1]))
        del frames, marks
    t_all1 = time.time()
    time.sleep(0.3)
    sampler.stop()
    assert eng.sync() == 0
    fill = math.ceil(B / T) if B > 0 else 0
    post = step_ms[fill + 1:]  # frames whose pool exceeds B
    first = fill + 2
    idx = list(range(first, first + len(post)))
    m = len(post)
    mx, my = sum(idx) / m, sum(post) / m
    var = sum((x - mx) ** 2 for x in idx)
    slope = sum((x - mx) * (y - my) for x, y in zip(idx, post)) / var if var > 0 else 0.0
    p50 = lambda xs: sorted(xs)[len(xs) // 2]
    clk = lambda w: sampler.summary(w[0], w[1], pad=0.0)["sm_mhz"]

    def pairs(n):  # visible (query, key) pairs per query head
        return T * (n - 1) * T + T * (T + 1) / 2

    def pairs_statekv(n):
        return T * min(B, (n - 1) * T) + T * (T + 1) / 2

    bins = []
    for b0 in range(1, N + 1, 32):
        b1 = min(N, b0 + 31)
        bins.append({"frames": f"{b0}..{b1}",
                     "p50_us": 1e3 * p50(step_ms[b0 - 1:b1]),
                     "sm_mhz": clk((wall[b0 - 1][0], wall[b1 - 1][1]))})
    line = {
        "curve": WORKLOAD_TEXT[args.workload],
        "state_capacity": B,
        "frames": N,
        "streams": S,
        "layers": L,
        "input_chunk_frames": chunk,
        "statekv_step_us_at": {str(n): 1e3 * step_ms[n - 1] for n in samples},
        "statekv_sm_mhz_at": {str(n): clk(wall[n - 1]) for n in samples},
        "full_attention_us_at": {str(n): 1e3 * full_ms[n] for n in samples},
        "full_attention_sm_mhz_at": {str(n): clk(full_wall[n]) for n in samples},
        "full_over_statekv_flops_at": {str(n): pairs(n) / pairs_statekv(n) for n in samples},
        "statekv_flatness": {
            "frames": f"{first}..{first + m - 1}",
            "p50_first32_us": 1e3 * p50(post[:32]),
            "p50_last_half_us": 1e3 * p50(post[m // 2:]),
            "slope_pct_per_100_frames": 100.0 * 100.0 * slope / my if my > 0 else None,
            "p50_all_us": 1e3 * p50(post),
        },
        "statekv_bins_of_32": bins,
        "clocks": sampler.summary(t_all0, t_all1),
        "note": "full attention = the attention call alone (the decode-cache append it also "
                "needs is the same as StateKV's and not included); StateKV = the whole step; "
                "sm_mhz = median nvidia-smi SM clock while the frames ran (nearest sample "
                "when none fell inside)",
    }
    print(json.dumps(line), flush=True)


def run_decode(args, local):
    """Decoding over the detailed cache after a prefilled video: one prompt of
    ``--prompt`` tokens, then single-token steps, each timed with CUDA events.
    The video's frames run first (untimed).  Prints one JSON line."""
    import torch

    from paper_2605_31598_gb300 import StateKV, make_config
    from paper_2605_31598_gb300.inputs import WORKLOADS, batch_qkv

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (no CPU fallback exists)")
    device = torch.device("cuda", local)
    torch.cuda.set_device(device)
    base = WORKLOADS[args.workload]
    N = args.frames or base.max_frames
    T, d = base.tokens_per_frame, base.head_dim
    steps = max(3, args.steps)
    extra = -(-(args.prompt + steps + 3) // T)
    shape = dataclasses.replace(base, max_frames=N + extra)
    S, L, Hq, Hkv = shape.num_streams, shape.num_layers, shape.num_q_heads, shape.num_kv_heads
    eng = StateKV(make_config(shape))
    out = None
    for n in range(1, N + 1):
        q, k, v = batch_qkv(shape, n, streams=range(S), layers=range(L), seed=args.seed,
                            device=device)
        out = out if out is not None else torch.empty_like(q)
        if eng.prefill_frame(q, k, v, out) != 0:
            raise RuntimeError(f"prefill failed at frame {n}")
    gen = torch.Generator(device="cpu").manual_seed(args.seed + 7)

    def tokens(n):
        mk = lambda h: (torch.randn((S, L, n, h, d), generator=gen) * d ** -0.5).to(
            torch.bfloat16).to(device)
        return mk(Hq), mk(Hkv), mk(Hkv)

    st = torch.cuda.current_stream()
    sampler = gpu_sampler(device)
    time.sleep(0.3)

    def timed(batch):
        """Runs decode steps back to back (inputs made beforehand), each
        bracketed by CUDA events; returns their times in ms and the wall
        window of the run."""
        outs = [torch.empty_like(q) for q, _, _ in batch]
        torch.cuda.synchronize()
        evs = []
        t0 = time.time()
        for (q, k, v), o in zip(batch, outs):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(st)
            rc = eng.decode_step(q, k, v, o)
            e1.record(st)
            if rc != 0:
                raise RuntimeError(f"statekv_decode_step returned {rc}")
            evs.append((e0, e1))
        torch.cuda.synchronize()
        return [a.elapsed_time(b) for a, b in evs], (t0, time.time())

    (prompt_ms,), _ = timed([tokens(args.prompt)])
    timed([tokens(1) for _ in range(3)])  # warm-up single-token steps
    tok, win = timed([tokens(1) for _ in range(steps)])
    tok_ms = sorted(tok)
    sampler.stop()
    assert eng.sync() == 0
    rows = N * T + args.prompt + 3 + steps // 2
    cache_bytes = S * L * Hkv * rows * d * 2 * 2  # K and V read once per token
    p50 = tok_ms[len(tok_ms) // 2]
    line = {
        "decode": WORKLOAD_TEXT[args.workload],
        "video_frames": N,
        "cache_rows_per_head": rows,
        "prompt_tokens": args.prompt,
        "prompt_us": 1e3 * prompt_ms,
        "token_p50_us": 1e3 * p50,
        "tokens_per_s": 1e3 / p50,
        "kv_read_gbs_at_p50": cache_bytes / (p50 * 1e-3) / 1e9,
        "kv_read_frac_of_hbm_at_p50": cache_bytes / (p50 * 1e-3) / 1e9 / peaks()[0],
        "clocks": sampler.summary(*win),
        "note": "one call = every (stream, layer); single tokens (<= 16 query rows per KV head) "
                "run the one-pass split-K decode kernel, which reads each K and V row once; the "
                "prompt runs the two-pass attention kernel",
    }
    print(json.dumps(line), flush=True)


def run_diagnostics(args, local):
    """App. A's assumption statistics on the full-attention baseline, on
    synthetic inputs of the workload's shape: every frame runs through the
    method (filling the decode cache); at sampled frames n the full-attention
    scores pass runs for frames n and n + 1 of every layer, then the
    concentration C_{n,B} (App. A.1) and the candidate-pool recall, weighted
    recall, retention and churn (App. A.2) for the paper's budgets.  Prints one
    JSON line with the means over sampled frames and layers and the device
    times of the passes."""
    import numpy as np
    import torch

    from paper_2605_31598_gb300 import StateKV, diagnostics, make_config
    from paper_2605_31598_gb300.inputs import WORKLOADS, batch_qkv

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (no CPU fallback exists)")
    device = torch.device("cuda", local)
    torch.cuda.set_device(device)
    base = WORKLOADS[args.workload]
    N = args.frames or 128
    shape = dataclasses.replace(base, max_frames=N + 1, num_streams=1)
    S, L, T = 1, shape.num_layers, shape.tokens_per_frame
    budgets = [1, 4, 16, 64, 256, 1024, 4096, 16384]
    sample = sorted({n for n in range(8, N, max(1, N // 8))} | {N - 1})
    eng = StateKV(make_config(shape))
    cap = shape.max_frames * T
    ws = torch.empty(eng.scores_workspace_bytes(), dtype=torch.uint8, device=device)
    st = torch.cuda.current_stream()
    conc, a2, t_scores, t_stats = [], {b: [] for b in budgets}, [], []

    def scores_of(q, k, v):
        sc = torch.empty((S, L, cap), dtype=torch.float32, device=device)
        out = torch.empty_like(q)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        if eng.full_attention_scores(q, k, v, out, sc, ws) != 0:
            raise RuntimeError("statekv_full_attention_scores failed")
        e1.record(st)
        torch.cuda.synchronize()
        t_scores.append(e0.elapsed_time(e1))
        return sc[0]

    prev = None
    for n in range(1, N + 1):
        q, k, v = batch_qkv(shape, n, streams=[0], layers=range(L), seed=args.seed, device=device)
        if n in sample or (n - 1) in sample:
            sc = scores_of(q, k, v)
            if n in sample:
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(st)
                conc.append(diagnostics.concentration(sc, (n - 1) * T, budgets))
                e1.record(st)
                torch.cuda.synchronize()
                t_stats.append(e0.elapsed_time(e1))
            if (n - 1) in sample and prev is not None:
                for b in budgets:
                    m = diagnostics.state_metrics(prev, sc, (n - 1) * T, T, b)
                    a2[b].append(np.stack([m["recall"], m["weighted_recall"], m["retention"],
                                           m["churn"]]))
            prev = sc if n in sample else None
        if eng.prefill_frame(q, k, v, torch.empty_like(q)) != 0:
            raise RuntimeError(f"prefill failed at frame {n}")
    assert eng.sync() == 0
    c = np.concatenate(conc)  # [frames * layers][budgets]
    line = {
        "diagnostics": WORKLOAD_TEXT[args.workload],
        "data": "synthetic (the values describe random inputs, not videos)",
        "frames": N, "sampled_frames": sample, "budgets": budgets,
        "concentration_mean": [float(x) for x in c.mean(axis=0)],
        "recall_mean": [float(np.mean([x[0] for x in a2[b]])) for b in budgets],
        "weighted_recall_mean": [float(np.mean([x[1] for x in a2[b]])) for b in budgets],
        "retention_mean": [float(np.mean([x[2] for x in a2[b]])) for b in budgets],
        "churn_mean": [float(np.mean([x[3] for x in a2[b]])) for b in budgets],
        "scores_pass_ms_last": t_scores[-1],
        "scores_pass_keys_last": (sample[-1] + 1) * T,
        "concentration_all_budgets_ms_last": t_stats[-1],
    }
    print(json.dumps(line), flush=True)


def run_block(args, local):
    """The full per-frame transformer block (synthetic random-init weights of
    the workload's layer widths, Qwen2-7B: hidden 3584, MLP 18944): every
    frame runs all layers in order -- RMSNorm, QKV projection + RoPE at the
    virtual positions, the StateKV step, output projection, SiLU MLP -- so
    the layers are sequential, as in a real model.  Times steady-state frames
    with CUDA events; the library's profile splits the time by kind.  Prints
    one JSON line."""
    import numpy as np
    import torch

    from paper_2605_31598_gb300 import StateKV, make_config
    from paper_2605_31598_gb300.inputs import BLOCKS, WORKLOADS, block_input, block_weights
    from paper_2605_31598_gb300.statekv import block_weights_array, statekv_block_config

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (no CPU fallback exists)")
    device = torch.device("cuda", local)
    torch.cuda.set_device(device)
    base = WORKLOADS[args.workload]
    S = args.streams or base.num_streams
    T, B, L = base.tokens_per_frame, base.state_capacity, base.num_layers
    Hq, Hkv, d = base.num_q_heads, base.num_kv_heads, base.head_dim
    fill = math.ceil(B / T) if B > 0 else 0
    steps = min(args.steps, 40)
    prof_steps = min(steps, 10)  # a second, profiled pass splits the time by kind
    nframes = fill + args.warmup + steps + prof_steps
    shape = dataclasses.replace(base, max_frames=nframes, num_streams=S)
    blk = BLOCKS["qwen7b"]
    H, I = blk.hidden, blk.intermediate
    eng = StateKV(make_config(shape))
    bc = statekv_block_config(H, I, blk.rms_eps, blk.rope_theta, 1.0, 0)
    wts = block_weights(shape, blk, device=device)
    warr = block_weights_array(wts)
    ws = torch.empty(eng.block_workspace_bytes(bc), dtype=torch.uint8, device=device)
    xs = [block_input(shape, blk, n, device=device) for n in range(1, nframes + 1)]
    y = torch.empty_like(xs[0])
    st = torch.cuda.current_stream()
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
    for n in range(fill + args.warmup):
        if eng.block_frame(bc, warr, xs[n], y, ws) != 0:
            raise RuntimeError(f"statekv_block_frame failed at frame {n + 1}")
    torch.cuda.synchronize()
    sampler = gpu_sampler(device)
    time.sleep(0.3)
    t0 = time.time()
    for i in range(steps):
        starts[i].record(st)
        if eng.block_frame(bc, warr, xs[fill + args.warmup + i], y, ws) != 0:
            raise RuntimeError("statekv_block_frame failed")
        ends[i].record(st)
    torch.cuda.synchronize()
    t1 = time.time()
    sampler.stop()
    ms = sorted(a.elapsed_time(b) for a, b in zip(starts, ends))
    p50 = ms[len(ms) // 2]
    # The by-kind split records events around every launch, which keeps
    # consecutive kernels from overlapping their launch with the previous
    # one's tail: it runs as a separate pass, and its frame time is reported
    # beside the unprofiled one.
    eng.profile(True)
    p0, p1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    p0.record(st)
    for i in range(prof_steps):
        if eng.block_frame(bc, warr, xs[fill + args.warmup + steps + i], y, ws) != 0:
            raise RuntimeError("statekv_block_frame failed")
    p1.record(st)
    torch.cuda.synchronize()
    prof = eng.profile_read()
    eng.profile(False)
    assert eng.sync() == 0
    per = lambda k: prof[k][1] / prof_steps
    weight_bytes = L * 2 * (H * (Hq + 2 * Hkv) * d + (Hq + 2 * Hkv) * d + H * Hq * d
                            + 2 * I * H + H * I)
    gemm_flops = 2 * S * T * L * (H * (Hq + 2 * Hkv) * d + H * Hq * d + 3 * I * H)
    attn_flops = L * S * 4 * d * Hq * (T * B + T * (T + 1) / 2)
    hbm, tf_burst, _, _ = peaks()
    line = {
        "block": WORKLOAD_TEXT[args.workload] + "; decoder layer: hidden 3584, MLP 18944, "
                 "QKV bias, RMSNorm, RoPE theta 1e6, SiLU MLP (synthetic random-init weights)",
        "streams": S,
        "frames_timed": steps,
        "p50_us_per_frame": 1e3 * p50,
        "frames_per_s": 1e3 / p50,
        "profiled_us_per_frame": 1e3 * p0.elapsed_time(p1) / prof_steps,
        "ms_per_frame_by_kind": {"projection_gemms": per(3), "attention_importance": per(1),
                                 "select_gather": per(2), "cache_append": per(0),
                                 "norm_rope_silu": per(4)},
        "gemm_weight_bytes_per_frame": weight_bytes,
        "gemm_weight_read_gbs": weight_bytes / (per(3) * 1e-3) / 1e9,
        "gemm_weight_read_frac_of_hbm": weight_bytes / (per(3) * 1e-3) / 1e9 / hbm,
        "gemm_tflops": gemm_flops / (per(3) * 1e-3) / 1e12,
        "attention_tflops": attn_flops / (per(1) * 1e-3) / 1e12,
        "clocks": sampler.summary(t0, t1),
        "note": "layers run in sequence (layer l+1 reads layer l's output); at one stream the "
                "projections read every weight once per frame for 196 rows, so they are "
                "bound by HBM bandwidth, not by the tensor cores",
    }
    print(json.dumps(line), flush=True)


SELECTIONS = {"importance": 0, "recency": 1, "layer": 2}
SELECTION_TEXT = {0: "top-B importance per KV head (the method)",
                  1: "recency window (baseline; no importance)",
                  2: "top-B of the layer-level importance, shared by the KV heads (App. A)"}


def main():
    ap = argparse.ArgumentParser(description=__doc__)
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", default=DEFAULT_WORKLOAD, choices=sorted(WORKLOAD_TEXT))
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--max-frames", type=int, default=0,
                    help="decode-cache capacity in frames (default: the workload's); "
                         "a small value keeps the arena small for profiler captures")
    ap.add_argument("--selection", choices=sorted(SELECTIONS), default="importance",
                    help="state policy: the method's top-B importance per KV head, the "
                         "recency-window baseline, or the layer-level top-B of App. A")
    ap.add_argument("--diagnostics", action="store_true",
                    help="App. A assumption statistics on the full-attention baseline")
    ap.add_argument("--block", action="store_true",
                    help="the full per-frame transformer block (all layers in sequence)")
    ap.add_argument("--streams", type=int, default=0,
                    help="--block: streams per call (default: the workload's)")
    ap.add_argument("--curve", action="store_true",
                    help="per-frame cost vs frame index, StateKV next to exact full attention")
    ap.add_argument("--frames", type=int, default=0, help="--curve: frames to run (default: "
                    "the workload's video length)")
    ap.add_argument("--capacity", type=int, default=None,
                    help="--curve: state capacity B in tokens (default: the workload's)")
    ap.add_argument("--decode", action="store_true",
                    help="decoding over the detailed cache after --frames video frames")
    ap.add_argument("--prompt", type=int, default=64, help="--decode: prompt tokens")
    args = ap.parse_args()
    if args.decode:
        run_decode(args, int(os.environ.get("LOCAL_RANK", 0)))
        return
    if args.curve:
        run_curve(args, int(os.environ.get("LOCAL_RANK", 0)))
        return
    if args.diagnostics:
        run_diagnostics(args, int(os.environ.get("LOCAL_RANK", 0)))
        return
    if args.block:
        run_block(args, int(os.environ.get("LOCAL_RANK", 0)))
        return
    if args.warmup < 3:
        raise SystemExit("--warmup must be at least 3")
    world, rank, local = dist_setup()
    if args.impl == "reference":
        run_reference(args, world, rank)
    else:
        run_ours(args, world, rank, local)
    if world > 1:
        import torch.distributed as dist

        dist.destroy_process_group()


if __name__ == "__main__":
    main()
