"""The work whose speed counts: block-causal attention as training, evaluation and
streaming programs call it, through the package's public entry points.

Kinds of case
  train   forward and backward of one attention layer through the autograd function
  eval    forward only (validation loss, full-window denoising), with or without LSE
  step    one streaming step: in-flight chunks against the ring, then the commit
  window  a pipelined window (sink anchor, re-shift, ring), then the commit of its oldest chunk
  qkv     the fused QKV projection's output split head-major, with temporal RoPE

Sizes are the model table's head layouts (B and L: 64 channels per head, 0.5B: 72, 1B
and 3B: 128), the repository's workloads and the small shapes of its tests.
"""
import math

import torch

import paper_2608_01127_gb300 as mw

BF16 = torch.bfloat16


def listed():
    return [
        # the smallest call: a toy window, as smoke tests and first steps of a user run it
        dict(name="eval_tiny_d64", kind="eval", B=1, H=2, d=64, n=4, T=64, gain=1.0, lse=True),
        # 3B layout, a short clip at an odd latent size (7 x 43 tokens per chunk)
        dict(name="eval_3b_odd", kind="eval", B=1, H=20, d=128, n=5, T=301, gain=1.0, lse=True),
        # full-window denoising of the 1B layout: 32 chunks of 600 tokens, no LSE needed
        dict(name="eval_1b_32x600", kind="eval", B=1, H=12, d=128, n=32, T=600, gain=1.0, lse=False),
        # L layout (16 heads of 64), a two-chunk clip: the short end of training
        dict(name="train_l_2x880", kind="train", B=1, H=16, d=64, n=2, T=880, gain=1.0),
        # B layout, 16 chunks of two latent frames: the usual training window
        dict(name="train_b12_d64", kind="train", B=2, H=12, d=64, n=16, T=880, gain=1.0),
        # 0.5B layout: 72 channels per head
        dict(name="train_05b_d72", kind="train", B=1, H=16, d=72, n=16, T=880, gain=1.0),
        # 16 heads of 128, 21 chunks, peaky logits as late in training: the largest
        dict(name="train_h16_d128_peaky", kind="train", B=1, H=16, d=128, n=21, T=880, gain=4.0),
        # a stream just begun: B layout, one committed chunk
        dict(name="step_start_d64", kind="step", B=1, H=12, d=64, W=1, T=880, ring=1, head=0),
        # steady streaming: one chunk against eight committed ones, the ring wraps
        dict(name="step_rolling_d128", kind="step", B=1, H=16, d=128, W=1, T=880, ring=8, head=5),
        # pipelined denoising: four in-flight chunks against twelve
        dict(name="step_pipelined_d128", kind="step", B=1, H=16, d=128, W=4, T=880, ring=12, head=7),
        # eight in-flight chunks, a one-frame sink turned by the evicted frames, twelve chunks
        dict(name="window_sink_rope_d128", kind="window", B=1, H=16, d=128, W=8, T=880, ring=12, head=3,
             sink=440, rope=32, shift=24),
        # the input side of a B-layout training step
        dict(name="qkv_rope_d64", kind="qkv", B=2, H=12, d=64, N=14080, rope=32, per_frame=440),
    ]


# ------------------------------------------------------------------ sizes and work

def _train_pairs(c):
    return c["B"] * c["H"] * c["T"] * c["T"] * c["n"] * (c["n"] + 1) // 2


def _ring_len(c):
    return c["ring"] * c["T"]


def _cache_pairs(c):
    W, T = c["W"], c["T"]
    return c["B"] * c["H"] * (W * T * (c.get("sink", 0) + _ring_len(c)) + T * T * W * (W + 1) // 2)


def work(case):
    c = case
    BH, d = c["B"] * c["H"], c["d"]
    if c["kind"] == "qkv":
        # every element read once and written once; six operations per rotated pair of Q and K
        return {"bytes": 2 * 3 * BH * c["N"] * d * 2, "flops": 2 * BH * c["N"] * (c["rope"] // 2) * 6}
    if c["kind"] == "train":
        rows = BH * c["n"] * c["T"]
        # Q, K, V, dO in; O, dQ, dK, dV out; LSE written by the forward and read by the backward
        return {"bytes": 8 * rows * d * 2 + 2 * rows * 4, "flops": 14 * d * _train_pairs(c)}
    if c["kind"] == "eval":
        rows = BH * c["n"] * c["T"]
        return {"bytes": 4 * rows * d * 2 + (rows * 4 if c["lse"] else 0), "flops": 4 * d * _train_pairs(c)}
    rows = BH * c["W"] * c["T"]
    keys = BH * (c.get("sink", 0) + _ring_len(c))
    commit = 2 * BH * c["T"] * d * 2  # written; its source is among the inputs
    return {"bytes": 4 * rows * d * 2 + rows * 4 + 2 * keys * d * 2 + commit,
            "flops": 4 * d * _cache_pairs(c)}


# ------------------------------------------------------------------ drawn cases

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["train", "train", "eval", "eval", "step", "step", "window", "qkv"])
        d = rng.choice([64, 64, 72, 128, 128, rng.choice([80, 88, 96, 112])])
        c = dict(kind=kind, B=rng.choice([1, 1, 1, 2]), H=rng.choice([12, 16, 20, rng.randint(1, 24)]), d=d)
        if kind == "qkv":
            c.update(N=_log_int(rng, 64, 20000), rope=rng.choice([0, 32, 2 * rng.randint(1, d // 2)]),
                     per_frame=_log_int(rng, 16, 600))
            if c["B"] * c["H"] * c["N"] * d > 2 * 12 * 14080 * 64 * 2:
                continue
        elif kind in ("train", "eval"):
            c.update(n=_log_int(rng, 1, 32), T=_log_int(rng, 64, 1100), gain=rng.choice([1.0, 1.0, 4.0]))
            if kind == "eval":
                c["lse"] = rng.random() < 0.5
        else:
            c.update(W=rng.choice([1, 1, 2, 4, 8]) if kind == "step" else rng.choice([2, 4, 8]),
                     T=_log_int(rng, 96, 1100), ring=rng.randint(1, 12))
            c["head"] = rng.randint(0, c["ring"])
            if kind == "window":
                c.update(sink=rng.choice([c["T"], (c["T"] + 1) // 2, 440]), rope=rng.choice([0, 32, 2 * rng.randint(1, d // 2)]),
                         shift=_log_int(rng, 1, 4000))
        if work(c)["flops"] <= most:
            return c


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator("cuda").manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)


def _inputs(c, seed):
    """The tensors a program has before the call, on the GPU."""
    g = _gen(seed)
    B, H, d = c["B"], c["H"], c["d"]
    if c["kind"] == "qkv":
        return {"qkv": _randn(g, B, c["N"], 3, H, d).to(BF16)}
    if c["kind"] in ("train", "eval"):
        shape = (B, H, c["n"] * c["T"], d)
        x = {n: _randn(g, *shape) for n in ("q", "k", "v")}
        if c["gain"] != 1.0:  # per-head gain on Q and K: from flat to peaky rows
            gain = 1.0 + (c["gain"] - 1.0) * torch.rand(H, generator=g, device="cuda").view(1, H, 1, 1)
            x["q"], x["k"] = x["q"] * gain, x["k"] * gain
        if c["kind"] == "train":
            x["do"] = _randn(g, *shape)
        return {n: t.to(BF16) for n, t in x.items()}
    # the ring has room for one chunk more than it holds, so that a step's commit fills a free
    # slot and evicts nothing: the same call can be repeated
    cap = _ring_len(c) + c["T"]
    x = {n: _randn(g, B, H, c["W"] * c["T"], d).to(BF16) for n in ("q", "k_new", "v_new")}
    x.update({n: _randn(g, B, H, cap, d).to(BF16) for n in ("k_ring", "v_ring")})
    if c["kind"] == "window":
        x.update({n: _randn(g, B, H, c["sink"], d).to(BF16) for n in ("k_sink", "v_sink")})
    return x


def prepare(case, seed):
    s = dict(case)
    s.update(_inputs(case, seed))
    if case["kind"] == "train":
        for n in ("q", "k", "v"):
            s[n].requires_grad_(True)
    if case["kind"] in ("step", "window"):
        # the ring's bookkeeping and the split workspace, kept for the whole stream
        s["cap"], s["len"] = s["k_ring"].shape[2], _ring_len(case)
        s["row0"] = case["head"] * case["T"]
        s["slot"] = mw.RingState(s["cap"], s["row0"], s["len"]).commit(case["T"])
        keys = case.get("sink", 0) + s["len"]
        nbytes = mw.mw_bca_cache_workspace_size(case["B"], case["H"], case["W"], case["T"], case["d"], keys)
        s["ws"] = torch.empty(max(nbytes, 256), dtype=torch.uint8, device="cuda")
    return s


# ------------------------------------------------------------------ one pass

def run(state):
    s = state
    T = s["T"] if "T" in s else 0
    if s["kind"] == "train":
        o = mw.BlockCausalAttention.apply(s["q"], s["k"], s["v"], T)
        dq, dk, dv = torch.autograd.grad(o, (s["q"], s["k"], s["v"]), s["do"])
        return {"o": o.detach(), "dq": dq, "dk": dk, "dv": dv}
    if s["kind"] == "eval":
        o, lse = mw.mw_bca_fwd(s["q"], s["k"], s["v"], T, need_lse=s["lse"])
        return {"o": o, "lse": lse}
    if s["kind"] == "step":
        o, lse = mw.mw_bca_cache_step(s["q"], s["k_new"], s["v_new"], s["k_ring"], s["v_ring"], s["row0"],
                                      s["len"], s["slot"], T, T, workspace=s["ws"])
        return {"o": o, "lse": lse, "k_ring": s["k_ring"], "v_ring": s["v_ring"]}
    if s["kind"] == "window":
        o, lse = mw.mw_bca_cache_fwd_rope(s["q"], s["k_new"], s["v_new"], s["k_sink"], s["v_sink"], s["k_ring"],
                                          s["v_ring"], s["row0"], s["len"], T, s["rope"], 10000.0, s["shift"],
                                          workspace=s["ws"])
        # the window's oldest chunk is done: its keys and values join the ring
        mw.mw_bca_cache_commit(s["k_ring"], s["v_ring"], s["slot"], s["k_new"][:, :, :T].contiguous(),
                               s["v_new"][:, :, :T].contiguous())
        return {"o": o, "lse": lse, "k_ring": s["k_ring"], "v_ring": s["v_ring"]}
    q, k, v = mw.mw_qkv_rope_split(s["qkv"], s["rope"], 10000.0, s["per_frame"], 0)
    return {"q": q, "k": k, "v": v}


# ------------------------------------------------------------------ the same in 64 bits

def _turn64(x, frames, rope):
    """Channel pairs (2i, 2i+1), i < rope / 2, turned by frame * 10000^(-2i / rope)."""
    if rope == 0:
        return x
    i = torch.arange(rope // 2, device=x.device, dtype=torch.float64)
    ang = frames.to(torch.float64)[:, None] * 10000.0 ** (-2.0 * i / rope)
    cos, sin = ang.cos(), ang.sin()
    y = x.clone()
    a, b = x[..., 0:rope:2], x[..., 1:rope:2]
    y[..., 0:rope:2] = a * cos - b * sin
    y[..., 1:rope:2] = a * sin + b * cos
    return y


def _rows64(q, k, v):
    """Plain softmax attention of the rows q over the keys k; the weights, O and LSE."""
    p = torch.matmul(q, k.transpose(-1, -2)) / math.sqrt(q.shape[-1])
    lse = torch.logsumexp(p, -1)
    p = p.sub_(lse[..., None]).exp_()
    return p, torch.matmul(p, v), lse


def exact(case, seed):
    c = case
    x = {n: t.to(torch.float64) for n, t in _inputs(c, seed).items()}
    if c["kind"] == "qkv":
        frames = torch.arange(c["N"], device="cuda") // c["per_frame"]
        q, k, v = (t.permute(0, 2, 1, 3) for t in x["qkv"].unbind(2))
        return {"q": _turn64(q, frames, c["rope"]), "k": _turn64(k, frames, c["rope"]), "v": v}
    T, sc = c["T"], 1.0 / math.sqrt(c["d"])
    if c["kind"] in ("train", "eval"):
        q, k, v = x["q"], x["k"], x["v"]
        o, lse = torch.empty_like(q), torch.empty_like(q[..., 0])
        train = c["kind"] == "train"
        if train:
            do, dq, dk, dv = x["do"], torch.empty_like(q), torch.zeros_like(k), torch.zeros_like(v)
        for j in range(c["n"]):
            own, seen = slice(j * T, (j + 1) * T), slice(0, (j + 1) * T)
            p, o[:, :, own], lse[:, :, own] = _rows64(q[:, :, own], k[:, :, seen], v[:, :, seen])
            if train:
                g = do[:, :, own]
                dv[:, :, seen] += torch.matmul(p.transpose(-1, -2), g)
                ds = torch.matmul(g, v[:, :, seen].transpose(-1, -2))
                ds -= (g * o[:, :, own]).sum(-1, keepdim=True)
                ds *= p
                dq[:, :, own] = torch.matmul(ds, k[:, :, seen]) * sc
                dk[:, :, seen] += torch.matmul(ds.transpose(-1, -2), q[:, :, own]) * sc
        if train:
            return {"o": o, "dq": dq, "dk": dk, "dv": dv}
        return {"o": o, "lse": lse if c["lse"] else None}
    cap, length = x["k_ring"].shape[2], _ring_len(c)
    at = (c["head"] * T + torch.arange(length + T, device="cuda")) % cap  # oldest first, then the free slot
    keys, values = x["k_ring"][:, :, at[:length]], x["v_ring"][:, :, at[:length]]
    if c["kind"] == "window":
        shift = torch.full((c["sink"],), c["shift"], device="cuda")
        keys = torch.cat([_turn64(x["k_sink"], shift, c["rope"]), keys], 2)
        values = torch.cat([x["v_sink"], values], 2)
    o, lse = torch.empty_like(x["q"]), torch.empty_like(x["q"][..., 0])
    for j in range(c["W"]):
        own, seen = slice(j * T, (j + 1) * T), slice(0, (j + 1) * T)
        _, o[:, :, own], lse[:, :, own] = _rows64(x["q"][:, :, own], torch.cat([keys, x["k_new"][:, :, seen]], 2),
                                                  torch.cat([values, x["v_new"][:, :, seen]], 2))
    x["k_ring"][:, :, at[length:]] = x["k_new"][:, :, :T]
    x["v_ring"][:, :, at[length:]] = x["v_new"][:, :, :T]
    return {"o": o, "lse": lse, "k_ring": x["k_ring"], "v_ring": x["v_ring"]}
