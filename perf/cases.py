"""Workloads of the hybrid attention operator as its users run it, for timing and for comparing two builds.

A case names an entry point (`call`), a geometry (batch, heads, head_dim, latent frames, patch rows and columns, chunk
and overlap in frames) and the options of the context.  Shapes come from the workload table of synth.py (the
Wan2.1-1.3B-shaped layers), from the tests' ragged geometries, or are generic.

Inputs follow synth.py: q, k, v ~ N(0, 1), q and k divided by their per-token per-head RMS where the block would have
normalised them already, phi parameters ~ N(0, 0.02^2), everything in the operator's data type.
"""
from __future__ import annotations

import math

import torch

from paper_2601_04342_b200 import binding, geometry

# call      forward: the whole sequence in one call on device tensors.  stream: the same sequence chunk by chunk.
#           host: the call that takes host tensors and copies inside.  static: the call that allocates nothing.
# layout    bhnd: [batch, heads, tokens, head_dim].  bnhd: token-major, as the block's projections write it.
# qk        the context normalises and rotates q and k itself (rms norm with weights, rotary tables).
# bidir     linear branch over all tokens outside the window (the form that is distilled first).
DEFAULTS = dict(call="forward", dtype="bf16", B=1, heads=12, d=128, T=21, H=30, W=52, chunk=3, overlap=1, layout="bhnd",
                qk=False, bidir=False, hidden=0, dim=0, P=2, layers=2, act="relu", c_mode="rowmax")


def _case(**kw):
    c = dict(DEFAULTS)
    c.update(kw)
    c["hidden"] = c["hidden"] or 2 * c["d"]
    c["dim"] = c["dim"] or 2 * c["d"]
    return c


def listed():
    return [
        # the smallest call: four frames of 8x8 patches in fp32, the precision one validates a model in
        _case(name="tiny_fp32", dtype="fp32", heads=2, d=64, T=4, H=8, W=8, chunk=1),
        # a caller with a fixed memory plan, on a ragged frame of 9x17 patches
        _case(name="static_small", call="static", heads=2, d=64, T=7, H=9, W=17),
        # a small ragged bf16 call: tiles end in the middle of frames, the last chunk is one frame
        _case(name="small_ragged", B=2, heads=4, T=7, H=9, W=17),
        # a layer of the 320x480 resolution (12,600 tokens) in fp32
        _case(name="fp32_320x480", dtype="fp32", H=20, W=30),
        # the same layer in bf16: what a device of limited memory runs
        _case(name="layer_320x480", H=20, W=30),
        # the layer of 81 frames of 480x832 video (32,760 tokens), the operator's main use
        _case(name="layer_480x832"),
        # that layer inside its block: token-major tensors, q and k normalised and rotated by the operator
        _case(name="block_480x832", layout="bnhd", qk=True),
        # classifier-free guidance on a longer video: two batch items of 63,960 tokens
        _case(name="cfg_long", B=2, T=41),
        # the layer chunk by chunk, as a streaming sampler or a caller short of memory runs it
        _case(name="stream_480x832", call="stream"),
        # heads of 64 channels, the other head size: 24 of them over the same tokens, one-frame chunks
        _case(name="heads_of_64", heads=24, d=64, chunk=1),
        # the form that is distilled first, with a deeper map of another degree and activation, two-frame chunks
        _case(name="bidir_deep_phi", bidir=True, H=20, W=32, chunk=2, P=3, dim=192, hidden=192, layers=3, act="softplus"),
        # the layer on tensors that live in pinned host memory
        _case(name="host_480x832", call="host"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any entry point, sizes over the listed cases' range, odd ones among them."""
    most = {"bf16": work(_case(B=2, T=41))["flops"], "fp32": work(_case(dtype="fp32", H=20, W=30))["flops"]}
    while True:
        c = _case(call=rng.choice(["forward"] * 5 + ["stream"] * 2 + ["host", "static"]),
                  dtype=rng.choice(["bf16"] * 4 + ["fp32"]), B=rng.choice([1, 1, 2]), d=rng.choice([128, 128, 64]),
                  heads=_log(rng, 1, 24), T=_log(rng, 2, 81), H=_log(rng, 5, 34), W=_log(rng, 8, 60),
                  chunk=rng.choice([1, 2, 3, 3, 4, 5, 7]), overlap=rng.choice([0, 1, 1, 2, 3]),
                  P=rng.choice([1, 2, 2, 2, 3, 4]), c_mode=rng.choice(["rowmax"] * 3 + ["zero"]))
        c["layout"] = rng.choice(["bhnd", "bnhd"]) if c["call"] in ("forward", "stream") else "bhnd"
        c["qk"] = c["call"] in ("forward", "stream") and rng.random() < 0.3
        c["bidir"] = c["call"] == "forward" and rng.random() < 0.2
        if c["P"] != 2 or rng.random() < 0.3:         # maps other than the default one
            c["dim"] = {3: rng.choice([96, 192]), 4: rng.choice([128, 256])}.get(c["P"], rng.choice([64, 128, 192, 256]))
            c["hidden"] = rng.choice([64, 96, 128, 192, 256])
            c["layers"] = rng.choice([2, 2, 3, 4])
            c["act"] = rng.choice(["relu", "relu", "softplus", "gelu"])
        chunks = -(-c["T"] // min(c["chunk"], c["T"]))
        per_chunk = min(c["chunk"], c["T"]) * c["H"] * c["W"]
        if c["call"] == "static":                      # what its fixed scratch holds (rehyat.h)
            bh, sd = c["B"] * c["heads"], c["d"] + 4
            if chunks > 16 or 2 * chunks * bh * c["dim"] * sd + bh * chunks * -(-per_chunk // 128) * 128 * sd > 1 << 21:
                continue
        if 64 <= c["T"] * c["H"] * c["W"] and work(c)["flops"] <= most[c["dtype"]] and work(c)["bytes"] <= 2 ** 31:
            return c


def _phi(c, gen, dtype):
    nh, d, Dh, Do = c["heads"], c["d"], c["hidden"], c["dim"]
    sizes = {"W1": (nh, Dh, d), "b1": (nh, Dh), "W2": (nh, Do, Dh), "b2": (nh, Do)}
    if c["layers"] > 2:
        sizes["Wmid"] = (nh, c["layers"] - 2, Dh, Dh)
        sizes["bmid"] = (nh, c["layers"] - 2, Dh)
    return {n: (0.02 * torch.randn(s, generator=gen, device="cuda")).to(dtype) for n, s in sizes.items()}


def prepare(case, seed):
    c = case
    dtype = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    HW, T = c["H"] * c["W"], c["T"]
    N = T * HW
    shape = (c["B"], c["heads"], N, c["d"]) if c["layout"] == "bhnd" else (c["B"], N, c["heads"], c["d"])
    s = {"c": c}
    for n in ("q", "k", "v"):
        x = torch.randn(shape, generator=gen, device="cuda")
        if n != "v" and not c["qk"]:
            x /= x.square().mean(-1, keepdim=True).sqrt_()
        s[n] = x.to(dtype)
        del x
    s["phi_q"], s["phi_k"] = _phi(c, gen, dtype), _phi(c, gen, dtype)
    if c["call"] != "static":
        s["op"] = binding.Rehyat(n_heads=c["heads"], head_dim=c["d"], dtype=c["dtype"], phi_hidden=c["hidden"], phi_dim=c["dim"],
                                 poly_degree=c["P"], act_hidden="relu" if c["act"] == "relu" else "gelu", act_out=c["act"],
                                 c_mode=c["c_mode"], max_batch=c["B"], max_tokens_per_frame=HW, max_chunk_frames=min(c["chunk"], T),
                                 bidirectional=c["bidir"], max_frames=T, phi_layers=c["layers"], qk_transform=c["qk"])
    if c["qk"]:
        w = [(1 + 0.1 * torch.randn((c["heads"], c["d"]), generator=gen, device="cuda")).to(dtype) for _ in range(2)]
        half = c["d"] // 2
        ang = torch.arange(N, device="cuda", dtype=torch.float64)[:, None] * \
            10000.0 ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half)[None, :]
        s["op"].set_qk_transform(q_weight=w[0], k_weight=w[1], cos=ang.cos().float(), sin=ang.sin().float())
    if c["call"] == "host":
        for n in ("q", "k", "v"):
            s[n] = s[n].cpu().pin_memory()
    # a streaming caller holds one output tensor and fills it chunk by chunk; the host and static calls want `out`
    if c["call"] == "host":
        s["out"] = torch.empty_like(s["q"], pin_memory=True)
    elif c["call"] in ("stream", "static"):
        s["out"] = torch.empty_like(s["q"])
    return s


def run(state):
    s, c = state, state["c"]
    geo = (c["T"], c["H"], c["W"], c["chunk"], c["overlap"])
    maps = (s["phi_q"], s["phi_k"])
    if c["call"] == "forward":
        return s["op"].forward(s["q"], s["k"], s["v"], *maps, *geo, layout=c["layout"])
    if c["call"] == "host":
        return s["op"].forward_host(s["q"], s["k"], s["v"], s["out"], *maps, *geo)
    if c["call"] == "static":
        act = "relu" if c["act"] == "relu" else "gelu"
        return binding.forward_static(s["q"], s["k"], s["v"], *maps, *geo, dtype=c["dtype"], poly_degree=c["P"],
                                      phi_hidden=c["hidden"], phi_dim=c["dim"], act_hidden=act, act_out=c["act"],
                                      c_mode=c["c_mode"], phi_layers=c["layers"], out=s["out"])
    # chunk by chunk: slices of the sequence, as [batch, heads, tokens, head_dim] views
    q, k, v, out = (t if c["layout"] == "bhnd" else t.transpose(1, 2) for t in (s["q"], s["k"], s["v"], s["out"]))
    HW = c["H"] * c["W"]
    s["op"].stream_begin(c["B"], c["H"], c["W"], min(c["chunk"], c["T"]), c["overlap"])
    for f0 in range(0, c["T"], c["chunk"]):
        f1 = min(f0 + c["chunk"], c["T"])
        sl = slice(f0 * HW, f1 * HW)
        s["op"].stream_step(q[:, :, sl], k[:, :, sl], v[:, :, sl], *maps, f1 - f0, out=out[:, :, sl])
    return s["out"]


def work(case):
    """Multiplications and additions of the method (softmax window, phi, state, read-out; no padding, nothing counted
    twice) and the bytes of q, k, v, out, the phi parameters and the rotation tables."""
    c = case
    HW, d, Dh, Do, mid = c["H"] * c["W"], c["d"], c["hidden"], c["dim"], c["layers"] - 2
    N, chunk = c["T"] * HW, min(c["chunk"], c["T"])
    bh = c["B"] * c["heads"]
    plan = geometry.chunk_plan(c["T"], HW, chunk, min(c["overlap"], c["T"]))
    if c["bidir"]:
        keys = N if len(plan) > 1 else 0
        queries = N if len(plan) > 1 else 0
    else:
        keys = plan[-1].lo
        queries = sum(p.q1 - p.q0 for p in plan if p.lo > 0)
    pairs = sum((p.q1 - p.q0) * (p.hi - p.lo) for p in plan)
    phi = 2 * (d * Dh + mid * Dh * Dh + Dh * Do)
    flops = bh * (4 * d * pairs + (phi + 2 * Do * (d + 1)) * (keys + queries))
    es = 2 if c["dtype"] == "bf16" else 4
    nbytes = es * (4 * bh * N * d + 2 * c["heads"] * (d * Dh + mid * Dh * (Dh + 1) + Dh * Do + Dh + Do))
    if c["qk"]:
        nbytes += 4 * N * d + 2 * es * c["heads"] * d
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # fp32: sums of up to some ten thousand terms in another order.  bf16: softmax weights, features and the output are
    # rounded to bf16 (2^-9 each); features taken to the power P carry P times that.
    return {"rel": 1e-5} if case["dtype"] == "fp32" else {"rel": 1e-2}
