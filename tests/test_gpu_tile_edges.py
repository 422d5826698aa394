"""Sizes at the edges of the kernels' own tiles, against the fp64 oracle through the C ABI (one B200)."""
import numpy as np
import pytest
import torch

from paper_2608_06838_b200 import binding, inputs
from paper_2608_06838_b200.inputs import Workload

from helpers import compare, oracle_reference, run_chain, tolerance
from test_gpu_variants import check, oracle_recurrent, run_recurrent

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# The warp-level kernels walk a block in tiles of 64 tokens (float32: 32) whatever the chunk: blocks shorter than a tile (3 chunks of 16),
# of one tile and a remainder (5 of 16, 3 of 32), of whole tiles; segments that end one token before, at and after a tile.
@pytest.mark.parametrize("chunk,cpb", [(16, 3), (16, 5), (32, 3), (64, 2), (64, 0)])
@pytest.mark.parametrize("dk,dv,dtype", [(32, 32, "f32"), (32, 64, "bf16"), (64, 64, "f32"), (64, 64, "bf16"), (128, 128, "f32")])
def test_cuda_core_tiles_and_blocks(dk, dv, dtype, chunk, cpb):
    w = Workload("tiles-%d-%d-%s-%d-%d" % (dk, dv, dtype, chunk, cpb), 2, 2, dk, dv, [129, 64, 63, 65, 1], chunk, dtype=dtype,
                 g_scale=0.1, s_in_sigma=0.3, ds_out_sigma=0.3, seed=61)
    x = inputs.make_inputs(w, DEV)
    got, _ = run_chain(w, x, chunks_per_block=cpb)
    compare(got, oracle_reference(x), tolerance(w), label=w.name)


@pytest.mark.parametrize("d,dtype", [(32, "f32"), (64, "f32"), (128, "f32"), (64, "bf16")])
def test_the_largest_finite_values(d, dtype):
    # the largest float32 (bf16 storage: the largest bf16) among the values and in the states: finite results stay finite
    w = Workload("largest-%d" % d, 1, 2, d, d, [100, 64], 32, dtype=dtype, g_scale=0.1, s_in_sigma=0.3, ds_out_sigma=0.003, seed=66)
    x = inputs.make_inputs(w, DEV)
    x["dO"] *= 0.01
    x["v"][0, 30, :, 1] = torch.finfo(x["v"].dtype).max
    x["v"][0, 31, :, 5] = -torch.finfo(x["v"].dtype).max
    x["S_in"][0, :, 3, 7] = torch.finfo(torch.float32).max
    got, _ = run_chain(w, x, chunks_per_block=2)
    compare(got, oracle_reference(x), tolerance(w), label=w.name)


@pytest.mark.parametrize("d,dtype,chunk", [(32, "f32", 16), (64, "f32", 64), (128, "f32", 32), (64, "bf16", 16), (32, "bf16", 64)])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_a_value_that_is_not_finite_reaches_no_token_that_does_not_depend_on_it(d, dtype, chunk, value):
    # o and dq of a token depend on v and k up to it, dk and dv on q and dO from it on
    w = Workload("nonfinite-%d-%s" % (d, dtype), 1, 2, d, d, [100, 77], chunk, dtype=dtype, g_scale=0.1, s_in_sigma=0.3, ds_out_sigma=0.3, seed=69)
    x = inputs.make_inputs(w, DEV)
    ref = oracle_reference(x)
    x["v"][0, 37, 0, 3] = value
    x["dO"][0, 50, 0, 2] = value
    got, _ = run_chain(w, x, chunks_per_block=2)
    clean = {n: slice(0, 37) for n in ("o", "dq")}
    clean.update({n: slice(51, None) for n in ("dk", "dv")})
    for n, s in clean.items():
        a, r = inputs.to_f64(got[n][0, s, 0]), ref[n][0, s, 0]
        assert np.isfinite(a).all() and np.abs(a - r).max() <= tolerance(w) * np.abs(ref[n]).max(), n
    assert not torch.isfinite(got["o"][0, 37, 0, 3]) and not torch.isfinite(got["dv"][0, 50, 0, 2])
    for n in ("o", "dq", "dk", "dv", "dg"):                      # the other head
        a = inputs.to_f64(got[n][0, :, 1])
        assert np.isfinite(a).all() and np.abs(a - ref[n][0, :, 1]).max() <= tolerance(w) * np.abs(ref[n]).max(), n


MASKS = [float("-inf"), torch.finfo(torch.float32).min, -1e30, -1e15]


@pytest.mark.parametrize("d,dtype,chunk", [(32, "f32", 16), (64, "f32", 64), (128, "f32", 32), (64, "bf16", 16), (32, "bf16", 64)])
def test_log_decays_that_mask(d, dtype, chunk):
    # a mask value wipes the state and no more: the weights of the tokens behind it, in the same tile, keep their own decays
    w = Workload("mask-%d-%s" % (d, dtype), 1, len(MASKS), d, d, [100, 77], chunk, dtype=dtype, g_scale=0.1, s_in_sigma=0.3, ds_out_sigma=0.3, seed=67)
    x = inputs.make_inputs(w, DEV)
    for h, m in enumerate(MASKS):
        for t in (0, 21, 22, 64, 117, 140 + h):
            x["g"][0, t, h] = m
    got, _ = run_chain(w, x, chunks_per_block=2)
    compare(got, oracle_reference(x), tolerance(w), label=w.name)


@pytest.mark.parametrize("chunk", [16, 32])
def test_chunked_delta_rule_with_log_decays_that_mask(chunk):
    w = Workload("delta-mask-%d" % chunk, 1, len(MASKS), 64, 32, [100, 77], chunk, dtype="f32", g_scale=0.1, s_in_sigma=0.5, ds_out_sigma=0.5, seed=68)
    x = inputs.make_variant_inputs(w, DEV)
    for h, m in enumerate(MASKS):
        for t in (0, 21, 22, 64, 117, 140 + h):
            x["g"][0, t, h] = m
    check(run_recurrent("delta_chunked", w, x), oracle_recurrent("delta", x), w.name)


# The chunkwise operators walk tiles of 32 tokens whatever the chunk: segments that end one token before, at and after a
# tile, inside its first four-token block, one token, and the shapes no other test runs.  24 heads take the delta rule's
# 16-column state pass (more than 148 CTAs with 8 columns).
@pytest.mark.parametrize("kind", ["delta", "channel"])
@pytest.mark.parametrize("dk,dv,chunk,H", [(128, 32, 32, 2), (128, 64, 32, 2), (32, 128, 32, 2), (64, 128, 16, 2), (64, 64, 32, 24),
                                           (128, 128, 16, 12)])
def test_chunked_operator_tiles(kind, dk, dv, chunk, H):
    w = Workload("%s-tiles-%d-%d-%d" % (kind, dk, dv, H), 1, H, dk, dv, [31, 32, 33, 3, 1, 100], chunk, dtype="f32", g_scale=0.3,
                 s_in_sigma=0.5, ds_out_sigma=0.5, seed=62)
    x = inputs.make_variant_inputs(w, DEV)
    check(run_recurrent(kind + "_chunked", w, x), oracle_recurrent(kind, x), w.name)


def test_chunked_diagonal_decay_with_wiped_channels():
    # channels that forget everything at some tokens: exponents down to -3000 inside a tile, every factor must stay finite
    w = Workload("channel-wipe", 1, 2, 64, 64, [100, 64], 32, dtype="f32", g_scale=0.05, s_in_sigma=0.5, ds_out_sigma=0.5, seed=64)
    x = inputs.make_variant_inputs(w, DEV)
    x["g_channel"][:, 37, :, ::3] = -100.0
    x["g_channel"][:, 40:70, :, 1] = -100.0
    check(run_recurrent("channel_chunked", w, x), oracle_recurrent("channel", x), w.name)


@pytest.mark.parametrize("kind", ["delta", "channel"])
@pytest.mark.parametrize("dtype,tol", [("f32", 1e-4), ("bf16", 2e-2)])
def test_chunked_operator_rows_without_vector_alignment(kind, dtype, tol):
    # rows one element apart from any 8- or 16-byte boundary: the entry points take them, the kernels load element by element
    w = Workload("%s-odd-%s" % (kind, dtype), 2, 2, 64, 32, [45], 32, dtype=dtype, g_scale=0.3, s_in_sigma=0.5, ds_out_sigma=0.5, seed=63)
    x = inputs.make_variant_inputs(w, DEV)
    ref = oracle_recurrent(kind, x)

    def odd(t):                                  # the same values with token rows of H*d + 1 elements, one element into the storage
        B, T, H, d = t.shape
        buf = torch.zeros(B * T * (H * d + 1) + 1, dtype=t.dtype, device=DEV)
        v = torch.as_strided(buf, t.shape, (T * (H * d + 1), H * d + 1, d, 1), 1)
        v.copy_(t)
        return v

    for n in ("q", "k", "v", "dO", "g_channel"):
        x[n] = odd(x[n])
    q, k, v, dO, S_in, dS_out = (x[n] for n in ("q", "k", "v", "dO", "S_in", "dS_out"))
    d = binding.make_desc(q, v, x["g"], w.chunk)
    o, dv_, dq, dk_ = (odd(torch.zeros_like(t)) for t in (v, v, q, k))
    dbeta, S, dS = torch.empty_like(x["beta"]), torch.empty_like(S_in), torch.empty_like(S_in)
    if kind == "delta":
        dg = torch.empty_like(x["g"])
        ws = torch.empty(binding.sf_delta_chunked_workspace_bytes(d, 1), dtype=torch.uint8, device=DEV)
        binding.sf_delta_chunked_fwd(d, q, k, v, x["g"], x["beta"], S_in, o, S, ws)
        binding.sf_delta_chunked_bwd(d, q, k, v, x["g"], x["beta"], S_in, dO, dS_out, dq, dk_, dv_, dg, dbeta, dS, ws)
    else:
        dg = odd(torch.zeros_like(x["g_channel"]))
        ws = torch.empty(binding.sf_channel_chunked_workspace_bytes(d, 1), dtype=torch.uint8, device=DEV)
        binding.sf_channel_chunked_fwd(d, q, k, v, x["g_channel"], S_in, o, S, ws)
        binding.sf_channel_chunked_bwd(d, q, k, v, x["g_channel"], S_in, dO, dS_out, dq, dk_, dv_, dg, dS, ws)
    torch.cuda.synchronize()
    check(dict(o=o, S_out=S, dq=dq, dk=dk_, dv=dv_, dg=dg, dbeta=dbeta, dS_in=dS), ref, w.name, tol)


# Tensor-core segments of one block start from the boundary state itself (no aggregate, no scan): one token, one chunk and its
# neighbours, longer ones by request; boundary states present and absent.
@pytest.mark.parametrize("L,cpb", [(1, 0), (63, 0), (64, 0), (65, 0), (500, 8), (512, 8), (1100, 18)])
@pytest.mark.parametrize("states", [True, False])
@pytest.mark.parametrize("saved", [True, False])
def test_one_block_segments(L, cpb, states, saved):
    w = Workload("one-block-%d" % L, 2, 3, 128, 128, [L], 64, g_scale=0.1, s_in_sigma=0.3 if states else None,
                 ds_out_sigma=0.3 if states else None, seed=65)
    x = inputs.make_inputs(w, DEV)
    d = binding.make_desc(x["q"], x["v"], x["g"], 64, cpb)
    assert binding.sf_num_blocks(d) == 1
    o, dq, dk, dv, dg = (torch.empty_like(x[n]) for n in ("v", "q", "k", "v", "g"))
    S, dS = (torch.empty(w.B, w.H, 128, 128, device=DEV) for _ in range(2))
    ws_f = torch.empty(binding.sf_workspace_bytes(d, 0), dtype=torch.uint8, device=DEV)
    ws_b = torch.empty(binding.sf_workspace_bytes(d, 1 if saved else 2), dtype=torch.uint8, device=DEV)
    binding.sf_segment_fwd(d, x["q"], x["k"], x["v"], x["g"], x["S_in"], o, S, ws_f)
    binding.sf_segment_bwd(d, x["q"], x["k"], x["v"], x["g"], x["S_in"], x["dO"], x["dS_out"], dq, dk, dv, dg, dS, ws_f if saved else None, ws_b)
    torch.cuda.synchronize()
    assert binding.sf_device_status() == 0
    compare(dict(o=o, S_out=S, dq=dq, dk=dk, dv=dv, dg=dg, dS_in=dS), oracle_reference(x), tolerance(w), label=w.name)


@pytest.mark.parametrize("C", [64, 33])                  # two channels per thread, one
def test_convolution_weight_gradient_with_infinite_last_inputs(C):
    # x_t meets dy_{t+j} under tap j: the last input only tap 0, the one before it taps 0 and 1
    B, L, W = 2, 70, 4
    gen = torch.Generator(device=DEV).manual_seed(70)
    x, dy, w = (torch.randn(*s, generator=gen, device=DEV) for s in ((B, L, C), (B, L, C), (W, C)))
    clean = x.clone()
    x[0, L - 1, 3] = float("inf")
    x[1, L - 2, 5] = float("nan")
    out = []
    for v in (clean, x):
        dx, dw, dtail = torch.empty_like(x), torch.empty_like(w), torch.empty(B, W - 1, C, device=DEV)
        binding.sf_conv_segment_bwd(v, w, None, dy, None, dx, dw, dtail)
        out.append(dw)
    torch.cuda.synchronize()
    ref, got = out
    assert not torch.isfinite(got[0, 3]) and torch.isfinite(got[1:, 3]).all()
    assert torch.isnan(got[:2, 5]).all() and torch.isfinite(got[2:, 5]).all()
    rest = [c for c in range(C) if c not in (3, 5)]
    assert torch.equal(got[:, rest], ref[:, rest])


@pytest.mark.parametrize("segs,cpb", [
    ([64, 192, 64, 320], 0), ([64, 192, 64, 320], 3), ([64] * 7, 64), ([320, 64, 100], 5),        # segments that begin inside a tile, odd blocks
    ([1], 0), ([65], 0), ([127], 0), ([128], 0), ([129], 1), ([191], 1), ([193], 2), ([449], 7),      # ragged ends of one- and two-chunk tiles
])
@pytest.mark.parametrize("merged", [0, 1])
def test_tensor_core_tiles_of_one_and_two_chunks(segs, cpb, merged):
    w = Workload("tc-tiles", 2, 3, 128, 128, segs, 64, g_scale=0.1, s_in_sigma=0.1, ds_out_sigma=0.1, seed=sum(segs))
    x = inputs.make_inputs(w, DEV)
    binding.sf_set_tuning(dict(merge_launches=merged))
    try:
        got, run = run_chain(w, x, chunks_per_block=cpb)
        S = run.S_bounds.clone()
    finally:
        binding.sf_set_tuning(None)
    compare(got, oracle_reference(x), tolerance(w), label="tc-tiles")
    tok = 0
    for i, n in enumerate(segs[:-1]):                       # the state entering each later segment
        tok += n
        part = {m: (t[:, :tok] if t is not None and t.dim() >= 3 and t.shape[1] == w.T else t) for m, t in x.items()}
        ref = oracle_reference(part)["S_out"]
        assert np.abs(inputs.to_f64(S[i + 1]) - ref).max() <= tolerance(w) * np.abs(ref).max()


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_tensor_core_tiles_keep_values_that_are_not_finite_to_their_sixteen_tokens(value):
    # what the masked products multiply by 0 reaches no row outside the value's own step of 16 tokens (96 .. 111)
    w = Workload("tc-inf", 1, 2, 128, 128, [384], 64, g_scale=0.1, seed=3)
    x = inputs.make_inputs(w, DEV)
    x["v"][0, 100, 0, 5] = value
    x["dO"][0, 100, 1, 7] = value
    got, _ = run_chain(w, x)
    assert torch.isfinite(got["o"][0, :96, 0].float()).all() and not torch.isfinite(got["o"][0, 100:, 0, 5].float()).any()
    assert torch.isfinite(got["o"][0, :, 1].float()).all()
    for n in ("dk", "dv"):
        assert torch.isfinite(got[n][0, 112:, 1].float()).all(), n
    assert not torch.isfinite(got["dv"][0, :101, 1, 7].float()).any()


@pytest.mark.parametrize("mask", [-200.0, -1e4, -1e30])
def test_tensor_core_tiles_with_log_decays_that_mask(mask):
    w = Workload("tc-mask", 1, 2, 128, 128, [200], 64, g_scale=0.1, s_in_sigma=0.1, seed=4)
    x = inputs.make_inputs(w, DEV)
    x["g"][0, [30, 31, 90, 150]] = mask
    d = binding.make_desc(x["q"], x["v"], x["g"], 64)
    o, S = torch.empty_like(x["v"]), torch.empty(1, 2, 128, 128, device=DEV)
    ws = torch.empty(max(binding.sf_workspace_bytes(d, 0), 256), dtype=torch.uint8, device=DEV)
    binding.sf_segment_fwd(d, x["q"], x["k"], x["v"], x["g"], x["S_in"], o, S, ws)
    torch.cuda.synchronize()
    ref = oracle_reference(x)
    for got, n in ((o, "o"), (S, "S_out")):
        assert np.abs(inputs.to_f64(got) - ref[n]).max() <= tolerance(w) * np.abs(ref[n]).max(), n


@pytest.mark.parametrize("cpb", [0, 1, 2, 3])
@pytest.mark.parametrize("merged,save_states", [(0, True), (0, False), (1, True)])
def test_tensor_core_blocks_with_log_decays_that_mask(cpb, merged, save_states):
    # several blocks: their aggregates weigh the tokens too.  Masks on the first and the last token of a chunk, of a segment and of the
    # ragged end, on odd and even tokens, on neighbours.
    masks = MASKS + [-200.0]
    w = Workload("tc-mask-blocks", 1, len(masks), 128, 128, [448, 321], 64, g_scale=0.1, s_in_sigma=0.3, ds_out_sigma=0.3, seed=70)
    x = inputs.make_inputs(w, DEV)
    for h, m in enumerate(masks):
        for t in (0, 21, 22, 64, 127, 140 + h, 447, 500, 575, 700, 768):
            x["g"][0, t, h] = m
    binding.sf_set_tuning(dict(merge_launches=merged))
    try:
        got, run = run_chain(w, x, chunks_per_block=cpb, save_states=save_states)
        S = inputs.to_f64(run.S_bounds[1])
    finally:
        binding.sf_set_tuning(None)
    compare(got, oracle_reference(x), tolerance(w), label=w.name)
    ref = oracle_reference({n: (t[:, :448] if n in ("q", "k", "v", "g", "dO") else t) for n, t in x.items()})["S_out"]
    assert np.abs(S - ref).max() <= tolerance(w) * np.abs(ref).max()
