"""The work that users of this library give it, as measurable cases.

One pass of a case is one call (or one forward + backward pair of calls) through the binding, on inputs drawn as
paper_2608_06838_b200.inputs draws them.  Kinds:

  chain    segments handed one after the other through ChainRun, forward + backward: what a training step runs for one
           linear-recurrence layer.  "graph": the step is recorded once and replayed, else it is launched from the host.
  segment  sf_segment_fwd alone ("fwd": evaluation or a prefill that carries the state), or followed by sf_segment_bwd
           with the forward's workspace ("saved") or from recomputed states ("replay": full recomputation)
  delta    the gated delta rule in its chunkwise form, forward + backward
  channel  the diagonal decay in its chunkwise form, forward + backward
  conv     the short convolution with a carried tail, forward + backward

"segs" lists segment lengths as text: "4096*8" or "12288,10240,8192".
"""
import math

import torch

from paper_2608_06838_b200 import binding, inputs
from paper_2608_06838_b200.inputs import Workload

DEVICE = "cuda:0"


# ---- the cases ----------------------------------------------------------------------------------------------------

def _chain(name, H, segs, d_k=128, d_v=128, chunk=64, dtype="bf16", graph=True, s_in=False, ds_out=False, B=1, g_scale=1.0):
    c = {"kind": "chain", "B": B, "H": H, "d_k": d_k, "d_v": d_v, "segs": segs, "chunk": chunk, "dtype": dtype, "graph": graph,
         "s_in": s_in, "ds_out": ds_out, "g_scale": g_scale}
    return dict(c, name=name) if name else c


def _segment(name, mode, B, H, L, d_k=128, d_v=128, chunk=64, dtype="bf16", g_scale=1.0):
    c = {"kind": "segment", "mode": mode, "B": B, "H": H, "d_k": d_k, "d_v": d_v, "segs": str(L), "chunk": chunk, "dtype": dtype,
         "s_in": True, "ds_out": mode != "fwd", "g_scale": g_scale}
    return dict(c, name=name) if name else c


def _ext(name, kind, B, H, L, d_k=64, d_v=64, chunk=32, dtype="f32", g_scale=0.1):
    c = {"kind": kind, "B": B, "H": H, "d_k": d_k, "d_v": d_v, "segs": str(L), "chunk": chunk, "dtype": dtype, "s_in": True,
         "ds_out": True, "g_scale": g_scale}
    return dict(c, name=name) if name else c


def _conv(name, B, L, C, W):
    c = {"kind": "conv", "B": B, "L": L, "C": C, "W": W}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a training step of one layer on a long context: 256K tokens in 16 segments, the benchmark's default workload
        _chain("chain-256k", 32, "16384*16", ds_out=True),
        # the same on 64K tokens with the decreasing segment lengths of a hybrid-aware partition and an incoming state
        _chain("chain-64k-nonuniform", 32, "12288,10240,8192*3,6144*3", s_in=True),
        # 32K tokens, 16 heads, launched from the host as an eager training loop does
        _chain("chain-32k-eager", 16, "4096*8", graph=False),
        # many short segments: the hand-off of the state between them counts
        _chain("chain-128k-seg1024", 40, "1024*128"),
        # one segment forward with a carried state: evaluation, or a prefill
        _segment("segment-fwd-8k", "fwd", 1, 32, 8192),
        # the smallest calls: a few hundred tokens, no whole number of chunks
        _segment("segment-fwd-200", "fwd", 1, 16, 200),
        # forward + backward with full recomputation, batched, ragged length
        _segment("segment-3001-replay", "replay", 2, 16, 3001),
        # float32 mode at the models' head width (checking runs, float32 training)
        _chain("chain-f32-8k", 16, "4096,2048,2000", dtype="f32", graph=False, s_in=True, g_scale=0.1),
        # narrow heads in bf16
        _chain("chain-bf16-d64-16k", 16, "8192*2", d_k=64, d_v=64, graph=False, g_scale=0.1),
        # the other transition families on the benchmark's segment
        _ext("delta-16k", "delta", 1, 16, 16384),
        _ext("channel-16k", "channel", 1, 16, 16384),
        # the short convolution in front of such a layer, 16 x 64 channels
        _conv("conv-16k", 1, 16384, 1024, 4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MAX_TOKEN_HEADS = 262144 * 32          # of the largest listed chain


def _draw_segs(rng, T, chunk):
    """Segment lengths for about T tokens: uniform ones with a shorter (sometimes ragged) last one, or a hybrid-aware partition."""
    if rng.random() < 0.3 and T >= 2048:
        lens = binding.sf_partition_hybrid(T // 128 * 128, rng.randint(2, 8), 1.0, rng.choice([1e-5, 1e-4, 1e-3]), rng.choice([0.5, 1.0]))
        return ",".join(str(s) for s in lens)
    seg = max(chunk, _log(rng, 512, 16384) // 128 * 128)
    n, rest = divmod(T, seg)
    rest = rest if rng.random() < 0.3 else rest // chunk * chunk
    parts = (["%d*%d" % (seg, n)] if n else []) + ([str(rest)] if rest else [])
    return ",".join(parts) if parts else str(chunk)


def draw(rng):
    r = rng.random()
    coin = lambda: rng.random() < 0.5  # noqa: E731
    g_scale = rng.choice([1.0, 0.1, 0.01])
    if r < 0.35:
        H = rng.choice([8, 16, 24, 32, 40])
        T = min(_log(rng, 2048, 262144), MAX_TOKEN_HEADS // H)
        return _chain(None, H, _draw_segs(rng, T, 64), graph=coin(), s_in=coin(), ds_out=coin(), g_scale=g_scale)
    if r < 0.60:
        B, H = rng.choice([1, 1, 2, 4]), rng.choice([4, 8, 12, 16, 32, 40])
        return _segment(None, rng.choice(["fwd", "fwd", "saved", "replay"]), B, H, _log(rng, 1, 16384), g_scale=g_scale)
    if r < 0.75:
        dtype = rng.choice(["f32", "bf16"])
        d_k, d_v = rng.choice([(32, 32), (64, 64), (32, 64)] + ([(128, 128)] if dtype == "f32" else []))
        chunk = rng.choice([16, 32, 64, 64])
        T = _log(rng, 256, 16384)
        return _chain(None, rng.choice([2, 4, 8, 16, 32]), _draw_segs(rng, T, chunk), d_k=d_k, d_v=d_v, chunk=chunk, dtype=dtype, graph=coin(),
                      s_in=coin(), ds_out=coin(), g_scale=g_scale)
    if r < 0.90:
        d_k, d_v = rng.choice([(32, 32), (64, 64), (64, 64), (32, 64), (64, 32), (128, 128)])
        chunk = 16 if d_k == 128 else rng.choice([16, 32, 32])
        H = rng.choice([2, 4, 8, 16])
        return _ext(None, rng.choice(["delta", "channel"]), rng.choice([1, 1, 2]), H, _log(rng, 64, 16384), d_k=d_k, d_v=d_v, chunk=chunk,
                    dtype=rng.choice(["f32", "f32", "bf16"]), g_scale=rng.choice([1.0, 0.1, 0.01]))
    C = rng.choice([64, 255, 768, 1024, 1500, 2048, 4096])
    return _conv(None, rng.choice([1, 1, 2, 4]), _log(rng, 16, 32768), C, rng.choice([2, 3, 4, 4, 4, 8]))


# ---- what a user's program has before the call --------------------------------------------------------------------

def _seg_lens(segs):
    out = []
    for part in segs.split(","):
        n, _, times = part.partition("*")
        out += [int(n)] * (int(times) if times else 1)
    return out


def _workload(case, seed):
    return Workload("case", case["B"], case["H"], case["d_k"], case["d_v"], _seg_lens(case["segs"]), case["chunk"], dtype=case["dtype"],
                    qk_norm="l2", g_scale=case["g_scale"], s_in_sigma=0.02 if case["s_in"] else None,
                    ds_out_sigma=0.02 if case["ds_out"] else None, seed=seed)


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device=DEVICE)


def _conv_inputs(case, seed):
    B, L, C, W = case["B"], case["L"], case["C"], case["W"]
    gen = torch.Generator(device=DEVICE).manual_seed(seed)

    def randn(*shape):
        return torch.randn(*shape, generator=gen, device=DEVICE)

    return {"x": randn(B, L, C), "w": randn(W, C) / W ** 0.5, "tail": randn(B, W - 1, C), "dy": randn(B, L, C), "dtail": randn(B, W - 1, C)}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "conv":
        x = _conv_inputs(case, seed)
        out = {"y": torch.empty_like(x["x"]), "tail_out": torch.empty_like(x["tail"]), "dx": torch.empty_like(x["x"]),
               "dw": torch.empty_like(x["w"]), "dtail_in": torch.empty_like(x["tail"])}
        return {"case": case, "x": x, "out": out}
    w = _workload(case, seed)
    if kind == "chain":
        x = inputs.make_inputs(w, DEVICE)
        run = binding.ChainRun(x["q"], x["k"], x["v"], x["g"], x["dO"], w.seg_lens, w.chunk)
        if case["graph"]:
            side = torch.cuda.Stream()
            torch.cuda.synchronize()                  # the inputs were made on another stream
            run.capture(x["S_in"], x["dS_out"], stream=side)
            side.synchronize()
        return {"case": case, "x": x, "run": run}
    x = inputs.make_inputs(w, DEVICE)
    g = x["g"]
    if kind in ("delta", "channel"):
        # the two families' own inputs (inputs.make_variant_inputs draws them the same way, and the convolution's besides)
        gen = torch.Generator(device=DEVICE).manual_seed(seed * 16 + 7)
        if kind == "channel":
            x["g"] = -torch.nn.functional.softplus(torch.randn(w.B, w.T, w.H, w.d_k, generator=gen, device=DEVICE)) * w.g_scale
        else:
            x["beta"] = torch.sigmoid(torch.randn(w.B, w.T, w.H, generator=gen, device=DEVICE))
    d = binding.make_desc(x["q"], x["v"], g, w.chunk)
    out = {"o": torch.empty_like(x["v"]), "S_out": torch.empty(w.B, w.H, w.d_k, w.d_v, device=DEVICE)}
    if kind != "segment" or case["mode"] != "fwd":
        out.update(dq=torch.empty_like(x["q"]), dk=torch.empty_like(x["k"]), dv=torch.empty_like(x["v"]), dg=torch.empty_like(x["g"]),
                   dS_in=torch.empty_like(out["S_out"]))
    if kind == "delta":
        out["dbeta"] = torch.empty_like(x["beta"])
    size = {"segment": binding.sf_workspace_bytes, "delta": binding.sf_delta_chunked_workspace_bytes,
            "channel": binding.sf_channel_chunked_workspace_bytes}[kind]
    backward = {"fwd": None, "saved": 1, "replay": 2}[case["mode"]] if kind == "segment" else 1
    return {"case": case, "x": x, "d": d, "out": out, "ws_f": _bytes(size(d, 0)), "ws_b": None if backward is None else _bytes(size(d, backward))}


# ---- one pass -----------------------------------------------------------------------------------------------------

def run(state):
    case, x = state["case"], state["x"]
    kind = case["kind"]
    if kind == "chain":
        r = state["run"]
        if case["graph"]:
            r.replay()
        else:
            r.forward(x["S_in"])
            r.backward(x["dS_out"])
        return {"o": r.o, "S_bounds": r.S_bounds, "dq": r.dq, "dk": r.dk, "dv": r.dv, "dg": r.dg, "dS_init": r.dS_init}
    y = state["out"]
    if kind == "conv":
        binding.sf_conv_segment_fwd(x["x"], x["w"], x["tail"], y["y"], y["tail_out"])
        binding.sf_conv_segment_bwd(x["x"], x["w"], x["tail"], x["dy"], x["dtail"], y["dx"], y["dw"], y["dtail_in"])
        return y
    d, ws_f, ws_b = state["d"], state["ws_f"], state["ws_b"]
    if kind == "segment":
        binding.sf_segment_fwd(d, x["q"], x["k"], x["v"], x["g"], x["S_in"], y["o"], y["S_out"], ws_f)
        if case["mode"] != "fwd":
            binding.sf_segment_bwd(d, x["q"], x["k"], x["v"], x["g"], x["S_in"], x["dO"], x["dS_out"], y["dq"], y["dk"], y["dv"], y["dg"],
                                   y["dS_in"], ws_f if case["mode"] == "saved" else None, ws_b)
    elif kind == "delta":
        binding.sf_delta_chunked_fwd(d, x["q"], x["k"], x["v"], x["g"], x["beta"], x["S_in"], y["o"], y["S_out"], ws_f)
        binding.sf_delta_chunked_bwd(d, x["q"], x["k"], x["v"], x["g"], x["beta"], x["S_in"], x["dO"], x["dS_out"], y["dq"], y["dk"], y["dv"],
                                     y["dg"], y["dbeta"], y["dS_in"], ws_b)
    else:
        binding.sf_channel_chunked_fwd(d, x["q"], x["k"], x["v"], x["g"], x["S_in"], y["o"], y["S_out"], ws_f)
        binding.sf_channel_chunked_bwd(d, x["q"], x["k"], x["v"], x["g"], x["S_in"], x["dO"], x["dS_out"], y["dq"], y["dk"], y["dv"], y["dg"],
                                       y["dS_in"], ws_b)
    return y


# ---- what a pass cannot do without --------------------------------------------------------------------------------

def work(case):
    """Bytes: every input read once per direction, every output written once.  Operations: those of the token recurrence
    (its products over the d_k x d_v state), the fewest any form of it needs."""
    kind = case["kind"]
    if kind == "conv":
        n, tail, wt = case["B"] * case["L"] * case["C"], case["B"] * (case["W"] - 1) * case["C"], case["W"] * case["C"]
        return {"bytes": 4 * (5 * n + 6 * tail + 3 * wt), "flops": 6 * n * case["W"]}
    lens = _seg_lens(case["segs"])
    e = 2 if case["dtype"] == "bf16" else 4
    dk, dv = case["d_k"], case["d_v"]
    th = case["B"] * case["H"] * sum(lens)
    gate = 4 * (dk if kind == "channel" else 1) + (4 if kind == "delta" else 0)
    fwd = (2 * dk + 2 * dv) * e + gate                     # q, k, v and the gates in, o out
    bwd = (4 * dk + 3 * dv) * e + 2 * gate                 # q, k, v, dO and the gates in, dq, dk, dv and the gates' gradients out
    state = 4 * case["B"] * case["H"] * dk * dv
    products = {"chain": (2, 5), "segment": (2, 5), "delta": (3, 9), "channel": (2, 5)}[kind]
    backward = kind != "segment" or case["mode"] != "fwd"
    nbytes = th * (fwd + (bwd if backward else 0))
    nbytes += state * ((len(lens) + 1 if kind == "chain" else 1 + case["s_in"]) + ((2 + case["ds_out"]) if backward else 0))
    return {"bytes": nbytes, "flops": 2 * dk * dv * th * (products[0] + (products[1] if backward else 0))}


def tolerance(case):
    """Measured on segments of 4096 and 16384 tokens under log-decay scales 1, 0.1 and 0.01 (relative 2-norm / largest error):

    bf16, 128-wide heads, against float32 arithmetic on the same bits: o, dq, dk, dv 2.3e-3 - 2.7e-3 / 2.2e-2, states 1.7e-3 / 1.1e-2;
    dg 4e-3 - 9e-3 / 4e-2 with blocks of 16 chunks and 1.4e-2 - 2.2e-2 / 7e-2 with blocks of 64, because it is a running sum of
    differences of rounded dot products; two forms that round in different places are both that far off, hence 3e-2.
    float32 chains: the same sum shows 2.1e-5 / 7e-5 from one block length to another, everything else below 1e-6.
    delta, channel in float32: up to 8.6e-7 / 7.3e-6 against the fp64 oracle.  bf16 storage with float32 arithmetic: 1.7e-3 / 3.9e-3
    against the oracle, the rounding of the stored outputs.  conv: up to 5.4e-8 / 3.7e-7 against the oracle."""
    if case["kind"] == "conv":
        return {"rel": 3e-7, "max": 3e-6}
    if case["dtype"] == "bf16":
        return {"rel": 3e-2, "max": 0.2} if case["d_k"] == 128 and case["kind"] in ("chain", "segment") else {"rel": 4e-3, "max": 1.6e-2}
    return {"rel": 8e-5, "max": 3e-4} if case["kind"] == "chain" else {"rel": 5e-6, "max": 5e-5}
