#!/usr/bin/env python
"""Benchmark: fwd+bwd tokens/s per linear-recurrence layer (chained segments, bf16) on B200.

One "step" = sf_chain_fwd + sf_chain_bwd over the whole synthetic sequence of one configuration
(all segments, state and state-gradient hand-offs included).  Prints ONE JSON line.  The default workload is
configuration 4 (256K tokens in 16 segments of 16384, H = 32), the largest single-GPU configuration.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--config {2,3,4,5}] [--seg-len L]
  python bench.py --impl reference ...      times the fp64 CPU oracle on a bounded sample instead
  python bench.py --op {delta_chunked,channel_chunked,delta,channel,conv}   one extension operator instead of the chain

Multi-GPU: the path does not shard (replicas only): with --gpus N each rank runs the same workload on
its own GPU, no data-path collective; value = N * tokens / max-over-ranks time.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "fwd+bwd tokens/s per linear-recurrence layer"
UNIT = "tokens/s"
BYTES_PER_TOKEN_HEAD = 2828          # q,k,v,dO read once, o,dq,dk,dv written once (bf16, d=128), g and dg float32
# of the chunkwise form with full chunks, d = 128, chunk 64: forward 98304 + backward 245760 (the kernels run 589824: sweeps over tiles of 128
# tokens, dk and dv apart, block aggregates)
FLOPS_PER_TOKEN_HEAD = 344064
# algorithmic bytes per token*head of each kernel (its own inputs read once, its own outputs written once)
KERNEL_BYTES = {"agg_kv": 516, "agg_qdo": 516, "fwd_out": 1028, "dq": 1284, "dkdv": 1540}
# DRAM bytes per token*head of each kernel from the ncu capture of the small case (profiles/, 262144 token*heads per
# launch), scaled to a bench launch by the token*heads it processes (traffic grows in proportion)
KERNEL_NCU_TRAFFIC = {"agg_kv": (135.303e6 + 3.147e6) / 262144, "agg_qdo": (135.303e6 + 3.152e6) / 262144,
                      "fwd_out": (210.912e6 + 40.357e6) / 262144, "dq": (278.086e6 + 47.586e6) / 262144,
                      "dkdv": (285.313e6 + 107.338e6) / 262144}


def peaks():
    """(HBM GB/s, bf16 TFLOP/s sustained, source): the measured peaks of this machine's B200s, else the fallback figures."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), float(d.get("bf16_tflops_sustained", d.get("bf16_tflops", 1400.0))), "measured"
    return 6650.0, 1400.0, "fallback"


def copy_probe(device, nbytes=1 << 30, reps=5):
    """Device-to-device copy bandwidth of this machine right now (read + write bytes per second), so that a degraded
    box shows in the report next to the roofline's fixed denominator.  Uses the driver's copy, none of this library."""
    import torch
    a = torch.empty(nbytes, dtype=torch.uint8, device=device)
    b = torch.empty_like(a)
    b.copy_(a)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(reps):
        b.copy_(a)
    e1.record()
    torch.cuda.synchronize()
    return 2.0 * nbytes * reps / (e0.elapsed_time(e1) * 1e-3) / 1e9


class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi while the timed region runs."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.lines = []
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q,
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
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
        except Exception:
            self.proc.kill()
        sm, mx, reasons = [], [], set()
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for name, val in zip(["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"], f[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm),
                "window": "timed region plus the same steps kept running until 3 samples were taken"}


def max_over_ranks(x: float, dist, device) -> float:
    """Max of a per-rank scalar (the timing rule for replicas: the slowest rank sets the step time)."""
    if dist is None:
        return float(x)
    import torch
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_throughput(tokens_per_rank: int, world: int, ms_per_step: float) -> float:
    """Whole-job tokens/s of `world` independent replicas that each process tokens_per_rank per step."""
    return world * tokens_per_rank / (ms_per_step * 1e-3)


def pick_workload(args):
    from paper_2608_06838_b200 import inputs
    if getattr(args, "small", False):
        return inputs.Workload("small-8k", 1, 32, 128, 128, [8192], 64, s_in_sigma=0.02, ds_out_sigma=0.02)
    if args.config == 5:
        return inputs.sweep_config(args.seg_len)
    return inputs.configs()[args.config - 1]


def cpu_baseline(w, budget_tokens=2048):
    """The oracle as it stands on the host cores, on the first `budget_tokens` tokens of the workload (all heads)."""
    import numpy as np
    import oracle
    from paper_2608_06838_b200 import inputs
    import dataclasses
    ws = dataclasses.replace(w, seg_lens=[budget_tokens])
    x = inputs.make_inputs(ws, "cpu")
    f = inputs.to_f64
    q, k, v, g, dO = (f(x[n]) for n in ("q", "k", "v", "g", "dO"))
    t0 = time.perf_counter()
    oracle.segment_fwd(q, k, v, g, f(x["S_in"]))
    oracle.segment_bwd(q, k, v, g, f(x["S_in"]), dO, f(x["dS_out"]))
    dt = time.perf_counter() - t0
    return {"value": ws.B * budget_tokens / dt, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
            "sample": "first %d tokens of the workload, all %d heads, unsplit, fwd+bwd, %.1f s" % (budget_tokens, w.H, dt)}


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    w = pick_workload(args)
    import oracle
    oracle.build()
    vals = []
    total = args.warmup + args.steps
    budget = 4096 if total > 3 else 8192          # per step; the whole run stays within a minute or two
    for i in range(total):
        r = cpu_baseline(w, budget)
        if i >= args.warmup:
            vals.append(r)
    v = statistics.mean(x["value"] for x in vals)
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * w.B * budget / v, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": w.name, "B": w.B, "H": w.H, "d_k": w.d_k, "d_v": w.d_v, "T": w.T, "chunk": w.chunk},
        "cpu_baseline": {"value": v, "unit": UNIT, "cores": vals[-1]["cores"], "kind": "oracle", "sample": vals[-1]["sample"]},
        "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


# ---- extension operators (diagonal decay, gated delta rule, short convolution): their own measured line ------------
EXT_OPS = ["delta_chunked", "channel_chunked", "delta", "channel", "conv"]


def extension_workload(op):
    """One 16384-token segment, H = 16, d_k = d_v = 64, float32 (268 MB of q, k, v, dO: larger than L2); chunk 32 for
    the chunkwise operators.  The convolution runs over the same tokens with H*d_v = 1024 channels, width 4."""
    from paper_2608_06838_b200 import inputs
    return inputs.Workload("ext-16k-h16-d64", 1, 16, 64, 64, [16384], 32, dtype="f32", qk_norm="l2", g_scale=0.1,
                           s_in_sigma=0.02, ds_out_sigma=0.02, seed=7)


def extension_bytes(op, w):
    """Algorithmic bytes per token*head, fwd + bwd: every input read once per direction, every output written once."""
    e = 4
    if op == "conv":                     # per token*head: d_v channels; x, y, dy, dx float32 (x is read in both directions)
        return 5 * w.d_v * e
    qk, vv = w.d_k * e, w.d_v * e
    gate = (w.d_k * e if op.startswith("channel") else e) + (e if op.startswith("delta") else 0)      # g (+ beta)
    fwd = 2 * qk + vv + gate + vv
    bwd = 2 * qk + 2 * vv + gate + 2 * qk + vv + gate
    return fwd + bwd


def extension_step_fn(op, w, x, dev):
    """Allocates outputs and workspaces once; returns a function that runs one fwd + bwd of the operator."""
    import torch
    from paper_2608_06838_b200 import binding
    q, k, v, dO = x["q"], x["k"], x["v"], x["dO"]
    if op == "conv":
        cx, cw, cdy = x["conv_x"], x["conv_w"], x["conv_dy"]
        y, dx, dw = torch.empty_like(cx), torch.empty_like(cx), torch.empty_like(cw)
        tail_out, dtail_in = torch.empty_like(x["conv_tail"]), torch.empty_like(x["conv_tail"])

        def step():
            binding.sf_conv_segment_fwd(cx, cw, x["conv_tail"], y, tail_out)
            binding.sf_conv_segment_bwd(cx, cw, x["conv_tail"], cdy, x["conv_dtail"], dx, dw, dtail_in)
        return step, 2
    g = x["g_channel"] if op.startswith("channel") else x["g"]
    beta = x["beta"]
    d = binding.make_desc(q, v, x["g"], w.chunk)
    o, dq, dk, dv, dg, dbeta = (torch.empty_like(t) for t in (v, q, k, v, g, beta))
    S_out = torch.empty(w.B, w.H, w.d_k, w.d_v, device=dev)
    dS_in = torch.empty_like(S_out)
    nbytes = {"delta_chunked": lambda b: binding.sf_delta_chunked_workspace_bytes(d, b),
              "channel_chunked": lambda b: binding.sf_channel_chunked_workspace_bytes(d, b)}.get(
                  op, lambda b: binding.sf_recurrent_workspace_bytes(d) if b else 16)
    ws_f = torch.empty(max(nbytes(0), 16), dtype=torch.uint8, device=dev)
    ws_b = torch.empty(max(nbytes(1), 16), dtype=torch.uint8, device=dev)
    S_in, dS_out = x["S_in"], x["dS_out"]
    if op == "delta_chunked":
        def step():
            binding.sf_delta_chunked_fwd(d, q, k, v, g, beta, S_in, o, S_out, ws_f)
            binding.sf_delta_chunked_bwd(d, q, k, v, g, beta, S_in, dO, dS_out, dq, dk, dv, dg, dbeta, dS_in, ws_b)
    elif op == "channel_chunked":
        def step():
            binding.sf_channel_chunked_fwd(d, q, k, v, g, S_in, o, S_out, ws_f)
            binding.sf_channel_chunked_bwd(d, q, k, v, g, S_in, dO, dS_out, dq, dk, dv, dg, dS_in, ws_b)
    elif op == "delta":
        def step():
            binding.sf_delta_segment_fwd(d, q, k, v, g, beta, S_in, o, S_out)
            binding.sf_delta_segment_bwd(d, q, k, v, g, beta, S_in, dO, dS_out, dq, dk, dv, dg, dbeta, dS_in, ws_b)
    else:
        def step():
            binding.sf_channel_segment_fwd(d, q, k, v, g, S_in, o, S_out)
            binding.sf_channel_segment_bwd(d, q, k, v, g, S_in, dO, dS_out, dq, dk, dv, dg, dS_in, ws_b)
    return step, None


def extension_cpu_baseline(op, w, tokens=8192):
    """The numpy fp64 oracle of the operator on the first `tokens` tokens (all heads)."""
    import dataclasses
    from oracle import variants as V
    from paper_2608_06838_b200 import inputs
    ws = dataclasses.replace(w, seg_lens=[tokens])
    x = inputs.make_variant_inputs(ws, "cpu")
    f = inputs.to_f64
    t0 = time.perf_counter()
    if op == "conv":
        V.conv_fwd(f(x["conv_x"]), f(x["conv_w"]), f(x["conv_tail"]))
        V.conv_bwd(f(x["conv_x"]), f(x["conv_w"]), f(x["conv_tail"]), f(x["conv_dy"]), f(x["conv_dtail"]))
    elif op.startswith("channel"):
        a = [f(x[n]) for n in ("q", "k", "v", "g_channel", "S_in")]
        V.channel_fwd(*a)
        V.channel_bwd(*a, f(x["dO"]), f(x["dS_out"]))
    else:
        a = [f(x[n]) for n in ("q", "k", "v", "g", "beta", "S_in")]
        V.delta_fwd(*a)
        V.delta_bwd(*a, f(x["dO"]), f(x["dS_out"]))
    dt = time.perf_counter() - t0
    return {"value": ws.B * tokens / dt, "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": "first %d tokens, all %d heads, fwd+bwd, %.1f s (numpy, one thread drives it)" % (tokens, w.H, dt)}


def run_extension(args):
    """fwd + bwd of one extension operator on its stated workload: device time, HBM roofline fraction, oracle timing."""
    if int(os.environ.get("RANK", "0")) != 0:
        return
    import torch
    from paper_2608_06838_b200 import binding, inputs
    torch.cuda.set_device(0)
    dev = "cuda:0"
    binding.load()
    op = args.op
    w = extension_workload(op)
    x = inputs.make_variant_inputs(w, dev)
    step, fixed_launches = extension_step_fn(op, w, x, dev)
    torch.cuda.synchronize()
    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    sampler = ClockSampler(0)
    sampler.start()
    regions = []
    n0 = binding.sf_launch_count()
    for _ in range(args.repeats):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(args.steps):
            step()
        e1.record()
        torch.cuda.synchronize()
        regions.append(e0.elapsed_time(e1) / args.steps)
    launches = binding.sf_launch_count() - n0
    t_end = time.time() + 0.7
    while time.time() < t_end:              # keep the same load up until the clock sampler has a few samples
        step()
    torch.cuda.synchronize()
    clocks = sampler.stop()
    assert binding.sf_device_status() == 0
    ms = statistics.median(regions)
    tokens = w.B * w.T
    hbm, _, src = peaks()
    bth = extension_bytes(op, w)
    achieved = bth * tokens * w.H / (ms * 1e-3) / 1e9
    out = {"metric": "fwd+bwd tokens/s, extension operator %s" % op, "value": tokens / (ms * 1e-3), "unit": UNIT, "n_gpus": 1,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "f32", "data": "synthetic",
           "timed_regions": {"repeats": args.repeats, "ms_per_step_min": min(regions), "ms_per_step_max": max(regions)},
           "config": {"workload": w.name, "operator": op, "B": w.B, "H": w.H, "d_k": w.d_k, "d_v": w.d_v, "T": w.T,
                      "chunk": w.chunk if op.endswith("chunked") else None, "conv_width": 4 if op == "conv" else None,
                      "l2": "inputs (268 MB) exceed L2, no flush", "parallelism": "replicas only"},
           "clocks": clocks, "e2e": None, "gpu_launches": int(launches),
           "roofline": {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s", "peak_source": src, "frac": achieved / hbm,
                        "traffic": None, "note": "whole operator, fwd + bwd: %d algorithmic bytes per token*head / step time; "
                                                 "float32 CUDA-core kernels, not bound by HBM" % bth}}
    if not args.skip_cpu:
        out["cpu_baseline"] = extension_cpu_baseline(op, w)
    print(json.dumps(out))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--config", type=int, default=4, choices=[2, 3, 4, 5],
                    help="benchmark configuration; default 4 = 256K tokens, 16 segments of 16384, H = 32 (the largest one)")
    ap.add_argument("--repeats", type=int, default=5, help="how many times the K-step timed region is repeated (median reported)")
    ap.add_argument("--seg-len", type=int, default=4096, help="segment length of configuration 5")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-overlap", action="store_true")
    ap.add_argument("--chunks-per-block", type=int, default=0)
    ap.add_argument("--small", action="store_true",
                    help="profiling case: one 8192-token segment, H=32 (tensors still exceed L2); implies no e2e / cpu legs")
    ap.add_argument("--no-graph", dest="graph", action="store_false",
                    help="launch the chain from the host every step instead of replaying it as one CUDA graph "
                         "(sf_chain_graph_*)")
    ap.add_argument("--no-autotune", dest="autotune", action="store_false",
                    help="keep the library's model for the block length instead of timing the candidates first "
                         "(sf_chain_autotune; only used when --chunks-per-block is 0)")
    ap.add_argument("--merge-launches", action="store_true",
                    help="install the merged-launch schedule (every stage once over the whole chain) instead of searching")
    ap.add_argument("--op", default="chain", choices=["chain"] + EXT_OPS,
                    help="chain (default): the segment chain of the main path; else fwd+bwd of one extension operator on a "
                         "16384-token, H = 16, d = 64 float32 segment")
    ap.add_argument("--skip-e2e", action="store_true")
    ap.add_argument("--skip-cpu", action="store_true")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3) if args.impl == "ours" else args.warmup
    if args.small:
        args.skip_e2e = args.skip_cpu = True
    if args.impl == "reference":
        run_reference(args)
        return
    if args.op != "chain":
        run_extension(args)
        return

    import torch
    from paper_2608_06838_b200 import binding, inputs

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = "cuda:%d" % local
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device(dev))
    binding.load()

    w = pick_workload(args)
    x = inputs.make_inputs(w, dev)
    run = binding.ChainRun(x["q"], x["k"], x["v"], x["g"], x["dO"], w.seg_lens, w.chunk, args.chunks_per_block)
    overlap = not args.no_overlap

    # a graph cannot be recorded on the legacy default stream: that mode runs on a stream of its own (which does not
    # wait for the default stream, where the inputs were generated, by itself)
    torch.cuda.synchronize()
    work_stream = torch.cuda.Stream() if args.graph else torch.cuda.current_stream()

    # Profile-guided tuning (untimed preparation, like the graph capture below), both with the same margin rule.  First the
    # schedule of the chain driver (streams, how far the aggregates run ahead, merged launches) at the library's own block
    # length, then the block length under the schedule that was installed: the best block length depends on the schedule.
    tuned = None
    if args.merge_launches:
        binding.sf_set_tuning(dict(merge_launches=1))
        tuned = {"schedule": {"merge_launches": 1, "forced": True}}
    if args.autotune and overlap and args.graph and not args.merge_launches:
        with torch.cuda.stream(work_stream):
            t, t_ms, d_ms = run.autotune_schedule(x["S_in"], x["dS_out"], reps=10, margin=0.02)
        work_stream.synchronize()
        tuned = {"schedule": {"sweep_streams": t.sweep_streams, "agg_streams": t.agg_streams, "scan_group_tokens": t.scan_group_tokens,
                              "agg_inorder_ctas": t.agg_inorder_ctas, "agg_ahead": t.agg_ahead, "merge_launches": t.merge_launches,
                              "ms": round(t_ms, 4), "default_ms": round(d_ms, 4)}}
    if args.autotune and args.chunks_per_block == 0:
        # candidates are timed the way the step will run: as graph replays on the work stream, or launched from the host
        # with --no-graph
        cands = [0, 16, 22, 29, 32, 43, 52, 64]
        with torch.cuda.stream(work_stream):
            best, cand_ms = run.autotune(x["S_in"], x["dS_out"], cands, reps=10, overlap=overlap)
        work_stream.synchronize()
        # the library's own model (candidate 0) stays unless a candidate beats it by more than 2 % over the 10 repetitions:
        # smaller differences are noise, and a block length that changes from run to run makes runs incomparable
        model_ms = cand_ms[0]
        best_ms = cand_ms[cands.index(best)]
        if model_ms > 0 and model_ms <= 1.02 * best_ms:
            best = 0
        run.desc.chunks_per_block = best
        tuned = tuned or {}
        tuned.update({"candidates": cands, "ms": [round(v, 4) for v in cand_ms], "chosen": best,
                      "rule": "model unless > 2 % faster over 10 reps"})
    if args.graph:
        with torch.cuda.stream(work_stream):
            run.capture(x["S_in"], x["dS_out"], overlap=overlap)
        work_stream.synchronize()

    def step():
        if args.graph:
            run.replay()
        else:
            run.forward(x["S_in"], overlap=overlap)
            run.backward(x["dS_out"], overlap=overlap)

    def barrier():
        torch.cuda.synchronize()
        if dist is not None:
            dist.barrier()
            torch.cuda.synchronize()

    with torch.cuda.stream(work_stream):
        for _ in range(args.warmup):
            step()
    barrier()
    # Clock samples must come from the GPU under this load.  The timed region of a small workload lasts a few
    # milliseconds, shorter than nvidia-smi's sampling period, so rank 0 waits for the sampler's first line before
    # the region (the sampler is then running) and keeps the same steps going, untimed, after the region until three
    # samples have been taken under load.
    sampler = ClockSampler(local)
    if rank == 0:
        sampler.start()
        t_wait = time.perf_counter()
        while not sampler.lines and time.perf_counter() - t_wait < 3.0:
            time.sleep(0.02)
        sampler.lines.clear()
    # the K-step region is timed `repeats` times back to back (barrier and synchronize around each); the median region
    # gives the reported value, the spread is reported next to it
    region_ms = []
    launches = 0
    for rep in range(max(1, args.repeats)):
        n0 = binding.sf_launch_count()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        barrier()
        with torch.cuda.stream(work_stream):
            e0.record()
            for _ in range(args.steps):
                step()
            e1.record()
        barrier()
        region_ms.append(max_over_ranks(e0.elapsed_time(e1), dist, dev))
        launches = binding.sf_launch_count() - n0
    ms = statistics.median(region_ms)
    if rank == 0:
        t_wait = time.perf_counter()
        while len(sampler.lines) < 3 and time.perf_counter() - t_wait < 3.0:
            with torch.cuda.stream(work_stream):
                step()
            torch.cuda.synchronize()
    assert binding.sf_device_status() == 0, "a bounded device-side wait ran out"
    clocks = sampler.stop() if rank == 0 else None
    probe = copy_probe(dev) if rank == 0 else None
    ms_per_step = ms / args.steps
    tokens = w.B * w.T
    value = replica_throughput(tokens, world, ms_per_step)

    # ---- per-stage device times (second pass with the library's stage timers on) -------------------
    # (overlap off here: with the side streams on, a kernel's bracketed time would include waiting for SMs
    # that kernels of other streams hold; the whole-step number above keeps the overlap)
    stage = None
    if rank == 0:
        binding.sf_stage_timing(True)
        for _ in range(args.steps):
            run.forward(x["S_in"], overlap=False)
            run.backward(x["dS_out"], overlap=False)
        torch.cuda.synchronize()
        stage = binding.sf_stage_timing_read()
        binding.sf_stage_timing(False)

    # ---- end-to-end through the host-memory entry point ----------------------------------------------
    e2e = None
    if not args.skip_e2e:
        host = {n: (None if t is None else t.detach().to("cpu").pin_memory()) for n, t in x.items()}
        outs = {n: torch.empty_like(host[m]).pin_memory() for n, m in
                [("o", "v"), ("dq", "q"), ("dk", "k"), ("dv", "v"), ("dg", "g")]}
        S_final = torch.empty(w.B, w.H, w.d_k, w.d_v, dtype=torch.float32).pin_memory()
        dS_init = torch.empty_like(S_final).pin_memory()
        desc = binding.make_desc(host["q"], host["v"], host["g"], w.chunk, int(run.desc.chunks_per_block), seg_len=w.seg_lens[0])
        scratch = torch.empty(binding.sf_e2e_device_bytes(desc, w.seg_lens), dtype=torch.uint8, device=dev)

        def e2e_step():
            binding.sf_chain_fwd_bwd_host(desc, w.seg_lens, host["q"], host["k"], host["v"], host["g"], host["S_in"],
                                          host["dO"], host["dS_out"], outs["o"], S_final, outs["dq"], outs["dk"], outs["dv"],
                                          outs["dg"], dS_init, scratch)
        e2e_step()
        barrier()
        n_e2e = max(2, min(args.steps, 3))
        t0 = time.perf_counter()
        for _ in range(n_e2e):
            e2e_step()              # synchronises its stream before returning
        dt = time.perf_counter() - t0
        dt = max_over_ranks(dt, dist, dev)
        nb = lambda t: 0 if t is None else t.numel() * t.element_size()
        h2d = sum(nb(host[n]) for n in ("q", "k", "v", "g", "dO", "S_in", "dS_out"))
        d2h = sum(nb(t) for t in outs.values()) + nb(S_final) + nb(dS_init)
        # the host-buffer results against the device chain's results on the same inputs (first and last 4096 tokens of
        # every output, both boundary results); the two runs may use different block lengths, hence a tolerance: twice the parity bound
        worst = 0.0
        pairs = [(outs["o"], run.o), (outs["dq"], run.dq), (outs["dk"], run.dk), (outs["dv"], run.dv), (outs["dg"], run.dg)]
        for h, dres in pairs:
            for sl in (slice(0, 4096), slice(-4096, None)):
                a, b = h[:, sl].float(), dres[:, sl].float().cpu()
                worst = max(worst, float((a - b).abs().max() / b.abs().max().clamp_min(1e-30)))
        for h, dres in ((S_final, run.S_bounds[-1]), (dS_init, run.dS_init)):
            b = dres.float().cpu()
            worst = max(worst, float((h - b).abs().max() / b.abs().max().clamp_min(1e-30)))
        assert worst <= 4e-2, "host-buffer entry point disagrees with the device chain: %.3e" % worst
        e2e = {"value": world * tokens * n_e2e / dt, "unit": UNIT, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
               "ms_per_step": 1e3 * dt / n_e2e, "max_norm_diff_vs_device_chain": worst}
        del scratch

    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return

    peak, tf_peak, peak_kind = peaks()
    roof = None
    # which roofline binds is derived, not asserted: time at the bf16 peak for the algorithmic FLOPs against time at the
    # HBM peak for the algorithmic bytes (per token*head); the slower one is the bound
    t_flop = FLOPS_PER_TOKEN_HEAD / (tf_peak * 1e12)
    t_byte = BYTES_PER_TOKEN_HEAD / (peak * 1e9)
    bound = "hbm" if t_byte >= t_flop else "tensor"
    path_roof = {"bound": bound, "achieved": BYTES_PER_TOKEN_HEAD * tokens * w.H / (ms_per_step * 1e-3) / 1e9, "peak": peak,
                 "unit": "GB/s", "peak_source": peak_kind,
                 "flop_time_over_byte_time": t_flop / t_byte,
                 "note": "whole step: 2828 algorithmic bytes per token*head / step time; %d FLOPs per token*head at the "
                         "sustained bf16 peak take %.2f of the time the bytes take at the HBM peak" % (FLOPS_PER_TOKEN_HEAD, t_flop / t_byte)}
    path_roof["frac"] = path_roof["achieved"] / peak
    if stage:
        heavy = [st for st in stage if st["name"] in KERNEL_BYTES and st["launches"]]
        dom = max(heavy, key=lambda st: st["ms"])
        per_launch_ms = dom["ms"] / max(dom["launches"], 1)
        # token*heads of the mean launch: one launch per segment, or one per step when the launches are merged
        th_per_launch = tokens * w.H * args.steps / max(dom["launches"], 1)
        alg = KERNEL_BYTES[dom["name"]] * th_per_launch
        traffic = KERNEL_NCU_TRAFFIC[dom["name"]] * th_per_launch if dom["name"] in KERNEL_NCU_TRAFFIC else None
        roof = {"bound": "hbm", "kernel": dom["name"], "achieved": alg / (per_launch_ms * 1e-3) / 1e9,
                "peak": peak, "unit": "GB/s", "peak_source": peak_kind, "traffic": traffic,
                "avg_launch_ms": per_launch_ms, "launches": dom["launches"],
                "note": "stage timers: second pass of the same steps at the same block length with the stream overlap off"}
        roof["frac"] = roof["achieved"] / peak
    # bounded CPU sample: about 5-10 s of oracle work on the machine's cores (fp64 copies of the sample: a few GB of host memory)
    cpu = None if args.skip_cpu else cpu_baseline(w, min(w.T, (49152 * 32 // w.H) // w.chunk * w.chunk))   # about 10 s of CPU work
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
        "data": "synthetic",
        "timed_regions": {"repeats": len(region_ms), "ms_per_step_median": ms_per_step,
                          "ms_per_step_min": min(region_ms) / args.steps, "ms_per_step_max": max(region_ms) / args.steps},
        "config": {"workload": w.name, "B": w.B, "H": w.H, "d_k": w.d_k, "d_v": w.d_v, "T": w.T, "segments": w.seg_lens,
                   "chunk": w.chunk, "chunks_per_block": args.chunks_per_block or (tuned.get("chosen", "auto") if tuned else "auto"),
                   "autotune": tuned, "overlap": overlap, "graph": bool(args.graph),
                   "l2": "inputs (%.0f MB) exceed L2, no flush" % (4 * tokens * w.H * w.d_k * 2 / 1e6),
                   "parallelism": "replicas only"},
        "clocks": clocks, "copy_probe_gbs": probe, "e2e": e2e, "gpu_launches": launches, "roofline": roof, "path_roofline": path_roof,
        "stages": stage, "cpu_baseline": cpu,
    }
    print(json.dumps(out))
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
