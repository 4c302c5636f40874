"""The work a user of this library has it do, as a list of cases that can be timed and compared.

A case is one call pattern at one size.  `prepare` makes what a program holds before the call (tensors on
the GPU, the decode state, the projections of the random features), `run` is one pass through the Python
binding, `work` says what the pass cannot do without and `tolerance` how far two correct implementations
at the same precision may be apart.

Kinds of pass:
  causal   hybrid_attn: windowed softmax heads and causal linear heads of one layer, the prefill of a
           language model; with "state" it also exports the decode state
  self     hybrid_attn_self: the bidirectional layer of an encoder
  linear   causal_linear_attn carrying S and z from call to call (a long prompt fed in pieces)
  window   window_attn on every head
  decode   decode_step: one token for every sequence of the batch, in lock step
  ragged   decode_step_ragged: the same for sequences at positions of their own, some slots idle
"""
from __future__ import annotations

import math

import torch

from paper_2412_19829_b200 import binding as gf
from paper_2412_19829_b200 import synth


def _case(kind, B, H, N, d, w, dtype="bf16", bnhd=False, favor=False, state=False):
    """h0: windowed heads, 3 of 16 unless the kind has only one sort of head.  N: tokens of the call, or,
    for the decoding kinds, tokens absorbed before it."""
    h0 = {"linear": 0, "window": H}.get(kind, max(1, int(3 * H / 16 + 0.5)))
    return dict(kind=kind, B=B, H=H, N=N, d=d, w=w, h0=h0, dtype=dtype, bnhd=bnhd, favor=favor, state=state)


def listed():
    return [
        # the smallest layer in fp32, a unit test's or a toy model's: launches and host time
        dict(_case("causal", 1, 2, 256, 64, 32, dtype="f32"), name="tiny_f32"),
        # a small language model's batch in the storage type it is served in ...
        dict(_case("causal", 8, 12, 2048, 64, 128), name="gpt2s"),
        # ... and in fp32, where results are checked or a model was kept in fp32
        dict(_case("causal", 8, 12, 2048, 64, 128, dtype="f32"), name="gpt2s_f32"),
        # one long document: few (batch, head) chains, so that a chain has to be shared by several SMs
        dict(_case("causal", 1, 32, 32768, 128, 512), name="long32k"),
        # twice the length at half the head width, in the [B, N, H, d] order a projection writes
        dict(_case("causal", 1, 16, 65536, 64, 512, bnhd=True), name="long64k_bnhd"),
        # prefill of a serving batch, exporting the state that decoding goes on from: the largest call
        dict(_case("causal", 64, 16, 4096, 64, 256, state=True), name="prefill4k"),
        # the long document with positive random features instead of elu + 1
        dict(_case("causal", 1, 32, 32768, 128, 512, favor=True), name="favor32k"),
        # the bidirectional layer on a long document, and on a batch of images with an odd token count
        dict(_case("self", 1, 32, 32768, 128, 512), name="self32k"),
        dict(_case("self", 64, 12, 197, 64, 64, bnhd=True), name="self197"),
        # a prompt fed in ragged pieces, the linear state carried from piece to piece
        dict(_case("linear", 2, 13, 3001, 128, 1), name="linear_resume"),
        # decoding after the prefill, one step of the whole batch: launch and latency bound
        dict(_case("decode", 64, 16, 4096, 64, 256), name="decode64"),
        # continuous batching of a wide model: the state no longer fits the L2 cache
        dict(_case("ragged", 128, 32, 4096, 128, 512), name="ragged128"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: 1 to 128 sequences, 2 to 32 heads, up to 65 536 tokens, windows of
    16 to 512, both head sizes, layouts, storage types and feature maps."""
    kind = rng.choice(["causal"] * 4 + ["self"] * 2 + ["linear", "window", "decode", "ragged"])
    d = rng.choice([64, 128])
    w = _log_int(rng, 16, 512)
    bnhd = rng.random() < 0.35
    if kind in ("decode", "ragged"):
        return _case(kind, _log_int(rng, 1, 128), rng.choice([2, 4, 8, 12, 16, 24, 32]), _log_int(rng, 64, 8192), d, w,
                     dtype="f32" if rng.random() < 0.15 else "bf16")
    if kind == "causal" and rng.random() < 0.2:  # fp32 storage, at sizes up to the small language model's
        H, N = rng.choice([2, 4, 8, 12]), _log_int(rng, 64, 2048)
        room = 8 * 12 * 2048 * 64 // (H * N * d)
        return _case(kind, _log_int(rng, 1, max(1, min(8, room))), H, N, d, min(w, 128), dtype="f32", bnhd=bnhd)
    favor = kind in ("causal", "self") and rng.random() < 0.2
    most = 1 << (26 if favor or kind == "window" else 27)  # elements of one tensor: half of the largest listed ones
    H = rng.choice([4, 8, 12, 13, 16, 24, 32])
    N = min(_log_int(rng, 100, 65536), most // (H * d))
    B = _log_int(rng, 1, max(1, min(64, most // (H * N * d))))
    return _case(kind, B, H, N, d, w, bnhd=bnhd, favor=favor, state=kind == "causal" and rng.random() < 0.3)


def _normal(gen, shape, dtype, gain=1.0):
    x = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    return (x if gain == 1.0 else x.mul_(gain)).to(dtype)


def prepare(case, seed):
    """Queries, keys and values of unit scale, as a layer norm and a projection leave them (with random
    features: d^-1/4 of it, the scale at which they approximate the softmax kernel)."""
    c = case
    B, H, N, d, w, h0 = (c[k] for k in ("B", "H", "N", "d", "w", "h0"))
    dtype = synth.torch_dtype(c["dtype"])
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": c}
    if c["kind"] in ("decode", "ragged"):
        s["qkv"] = [_normal(gen, (B, H, d), dtype) for _ in range(3)]
        st = s["st"] = gf.DecodeState(B, H, d, w, h0, dtype)
        st.k_cache.copy_(_normal(gen, st.k_cache.shape, dtype))
        st.v_cache.copy_(_normal(gen, st.v_cache.shape, dtype))
        # sums over N tokens: phi of a unit normal has mean 1.16 and second moment about 1.7
        st.S.copy_(_normal(gen, st.S.shape, torch.float32, 1.3 * N**0.5))
        st.z.copy_(_normal(gen, st.z.shape, torch.float32, 0.6 * N**0.5).add_(1.16 * N))
        st.t = N
        if c["kind"] == "ragged":
            t = torch.randint(0, N + 1, (B,), generator=gen, device="cuda")
            idle = torch.rand(B, generator=gen, device="cuda") < 0.1
            s["t_seq"] = torch.where(idle, -torch.ones_like(t), t)
        return s
    shape = (B, N, H, d) if c["bnhd"] else (B, H, N, d)
    gain = d**-0.25 if c["favor"] else 1.0
    s["qkv"] = [_normal(gen, shape, dtype, gain if i < 2 else 1.0) for i in range(3)]
    s["layout"] = gf.GF_BNHD if c["bnhd"] else gf.GF_BHND
    s["W"] = synth.favor_projection(H - h0, d, seed=seed, dtype=c["dtype"]).cuda() if c["favor"] else None
    if c["state"]:
        s["st"] = gf.DecodeState(B, H, d, w, h0, dtype)
    if c["kind"] == "linear":
        s["S"] = torch.zeros(B, H, d, d, device="cuda")
        s["z"] = torch.zeros(B, H, d, device="cuda")
    return s


def run(s):
    c = s["case"]
    q, k, v = s["qkv"]
    kind, w, h0 = c["kind"], c["w"], c["h0"]
    if kind == "causal":
        st = s.get("st")
        o = gf.hybrid_attn(q, k, v, w, h0, layout=s["layout"], state_out=st, W=s["W"])
        return [o] if st is None else [o, st.k_cache, st.v_cache, st.S, st.z]
    if kind == "self":
        return [gf.hybrid_attn_self(q, k, v, w, h0, layout=s["layout"], W=s["W"])]
    if kind == "linear":
        return [gf.causal_linear_attn(q, k, v, s["S"], s["z"], layout=s["layout"]), s["S"], s["z"]]
    if kind == "window":
        return [gf.window_attn(q, k, v, w, layout=s["layout"])]
    st = s["st"]
    if kind == "decode":
        return [gf.decode_step(q, k, v, st), st.k_cache, st.v_cache, st.S, st.z]
    return [gf.decode_step_ragged(q, k, v, st, s["t_seq"]), st.k_cache, st.v_cache, st.S, st.z, s["t_seq"]]


def work(case):
    """Every input read once and every output written once; the products of Algorithm 1 token by token, the
    two products of the windowed heads over the visible keys, the projections of the random features."""
    c = case
    B, H, N, d, w, h0 = (c[k] for k in ("B", "H", "N", "d", "w", "h0"))
    h1, es = H - h0, 4 if c["dtype"] == "f32" else 2
    if c["kind"] in ("decode", "ragged"):
        keys = min(N + 1, w) if c["kind"] == "decode" else sum(min(N * (i + 0.5) / 64, w) for i in range(64)) / 64
        live = 1.0 if c["kind"] == "decode" else 0.9
        ring = 2 * h0 * (keys + 1) * d * es  # the visible keys and values read, one of each written
        state = 2 * h1 * (d * d + d) * 4
        return {"bytes": B * (4 * H * d * es + live * (ring + state)), "flops": B * live * (4 * h0 * keys * d + 4 * h1 * d * d)}
    nbytes = 4 * B * H * N * d * es
    we = min(w, N)
    seen = N * we - we * (we - 1) // 2  # pairs (query, visible key) of a causal window
    if c["kind"] == "self":
        seen = 2 * seen - N
    flops = B * (4 * h0 * seen * d + 4 * h1 * N * d * d)
    if c["favor"]:
        flops += 4 * B * h1 * N * d * d
        nbytes += h1 * d * d * es
    if c["state"]:
        nbytes += B * (2 * h0 * we * d * es + h1 * (d * d + d) * 4)
    if c["kind"] == "linear":
        nbytes += 2 * B * h1 * (d * d + d) * 4
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times what is seen against the same path in 64 bits.  fp32 sums: 2.3e-7 (largest element
    3e-6).  bf16: 2.6e-3, from the rounding of P and of the features; single elements are off by up to 0.17
    of the root mean square, which is small beside the first rows of a long sequence.  bf16 decoding: 1.7e-3
    (4e-3), the rounding of the output."""
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 1.5e-5}
    if case["kind"] in ("decode", "ragged"):
        return {"rel": 7e-3, "max": 2e-2}
    return {"rel": 1e-2, "max": 0.5}
