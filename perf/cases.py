"""The work that users of the library have it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``kind`` says what one pass is:

  prefill   a batch of prompts: lte_scores, lte_select, lte_attn_prefill and, with ``cache``, lte_cache_init
  decode    ``steps`` generated tokens for every sequence of a batch on top of the cache a prompt of T tokens left; with the
            three-layer scorer one lazy scoring of the ring as well
  chunk     T more prompt tokens arriving at a cache that holds ``past`` tokens (lte_attn_prefill_chunk)
  train     one layer's part of a training step: scores, selection, attention, the Eq. 7 statistics, backward

``scorer`` is "cnn" (one layer of K taps) or "stack" (the paper's three layers); with ``rope`` the cached keys carry a rotary
embedding, which the scorer must not see.  H counts key/value heads, G query heads per key/value head.  ``half`` gives the
scorer a bias for which about half of the budget R is in use, as in the paper's trained models; without it the budget binds.
Values and distributions are those of the benchmark configurations: q, k ~ N(0,1)/d^0.25, v, dO ~ N(0,1).
"""
import math
from statistics import NormalDist

import torch

from paper_2510_20787_b200 import lte

DTYPES = {"bf16": (torch.bfloat16, lte.BF16, 2), "f32": (torch.float32, lte.F32, 4)}


def _case(name, kind, dtype, B, H, G, T, d, W, R, sink=0, scorer="cnn", K=7, half=False, rope=False, cache=False, steps=0, past=0,
          streaming=False):
    c = {"kind": kind, "dtype": dtype, "B": B, "H": H, "G": G, "T": T, "d": d, "W": W, "R": R, "sink": sink, "scorer": scorer, "K": K,
         "half": half, "rope": rope, "cache": cache, "steps": steps, "past": past, "streaming": streaming}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call there is: configuration C1, fp32 (a unit test, a tiny model, a debugging session)
        _case("tiny fp32 prompt", "prefill", "f32", 1, 2, 1, 128, 32, 16, 8, K=5),
        # one user's short prompt of no round length, cached for the decode steps that follow: latency counts
        _case("one short prompt", "prefill", "bf16", 1, 16, 1, 777, 64, 128, 128, cache=True),
        # configuration C2, the headline prefill
        _case("prompt batch C2", "prefill", "bf16", 4, 16, 1, 4096, 64, 128, 128),
        # configuration C3, one long document at d = 128
        _case("long prompt C3", "prefill", "bf16", 1, 16, 1, 32768, 128, 512, 512),
        # the paper's serving shape: 32 query heads on 8, window 768, budget 512 half used, sink tokens, three-layer scorer on the keys
        # before their rotary embedding, 4K prompts, batch 32
        _case("serving prompts", "prefill", "bf16", 32, 8, 4, 4096, 64, 768, 512, sink=4, scorer="stack", half=True, rope=True, cache=True),
        # configuration C4: batched decode (the pool is full after the prompt)
        _case("decode C4", "decode", "bf16", 128, 16, 1, 2048, 64, 128, 128, steps=8),
        # decode of the paper's serving shape, with one lazy scoring per 64 tokens
        _case("serving decode", "decode", "bf16", 32, 8, 4, 2048, 64, 768, 512, sink=4, scorer="stack", half=True, rope=True, steps=64),
        # one user's answer after a long document at d = 128: latency counts
        _case("one answer d128", "decode", "bf16", 1, 16, 1, 2048, 128, 512, 512, steps=16),
        # the next 512 tokens of eight conversations
        _case("conversation turn", "chunk", "bf16", 8, 16, 1, 512, 64, 768, 512, past=2048),
        # configuration C5: training step
        _case("train C5", "train", "bf16", 8, 16, 1, 2048, 64, 64, 64),
        # training as the paper does it: three-layer scorer, its window and budget, grouped queries, the budget not binding
        _case("train three-layer scorer", "train", "bf16", 4, 8, 4, 4096, 64, 768, 512, sink=4, scorer="stack", half=True),
        # long-context training at d = 128 (heads and window of C3)
        _case("train long d128", "train", "bf16", 1, 16, 1, 8192, 128, 512, 512),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _cost(c):
    """Comparable size of a case; a training step takes about twice as long as a prefill with as many operations."""
    w = work(c)
    return max(w["bytes"], w["flops"] / 50) * {"prefill": 1, "decode": 2, "chunk": 2, "train": 2}[c["kind"]]


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["prefill", "prefill", "prefill f32", "decode", "decode", "chunk", "train", "train"])
        if kind == "prefill f32":
            c = _case(None, "prefill", "f32", rng.randint(1, 2), rng.randint(1, 4), 1, _log_int(rng, 64, 1024), 32, _log_int(rng, 8, 64),
                      _log_int(rng, 4, 64), K=5)
        else:
            stack = rng.random() < 0.4
            d = 64 if stack else rng.choice([64, 64, 128])
            W, R = _log_int(rng, 32, 768), _log_int(rng, 16, 512)
            c = _case(None, kind, "bf16", 1, rng.choice([8, 16]), rng.choice([1, 1, 4]), _log_int(rng, 256, 32768), d, W, R,
                      sink=rng.choice([0, 4]), scorer="stack" if stack else "cnn", K=rng.choice([5, 7, 7]), half=rng.random() < 0.5,
                      rope=stack and kind in ("prefill", "decode"), cache=kind == "prefill" and rng.random() < 0.5)
            c["B"] = _log_int(rng, 1, 128 if kind == "decode" else 32)
            if kind == "decode":
                c["T"] = _log_int(rng, 256, 2048)
                c["steps"] = min(64, W - 13) if stack else _log_int(rng, 4, 32)
            elif kind == "chunk":
                c["T"], c["past"] = _log_int(rng, 64, 4096), _log_int(rng, 256, 4096)
                c["streaming"] = rng.random() < 0.3
            elif kind == "train":
                c["T"] = _log_int(rng, 256, 8192)
        if _cost(c) <= most:
            return c


def _scorer(c, g, dev):
    d, H = c["d"], c["H"]
    if c["scorer"] == "cnn":
        w = torch.randn((H, c["K"], 2 * d), generator=g, device=dev) * (0.1 if c["dtype"] == "f32" else 0.05)
        return lambda bias: lte.conv(w, bias)
    ch = [2 * d, d, d // 2, d // 4]
    wl = [torch.randn((H, ch[i + 1], 3, ch[i]), generator=g, device=dev) * (1.5 / math.sqrt(3 * ch[i])) for i in range(3)]
    wout = torch.randn((H, ch[3]), generator=g, device=dev) * (2.0 / math.sqrt(ch[3]))
    return lambda bias: lte.conv_stack(wl, wout, bout=bias)


def _rotated(k, cos, sin):
    """Rotary embedding of k [..., T, d] at positions 0 .. T-1 (half-split pairs)."""
    T, h = k.shape[-2], k.shape[-1] // 2
    x1, x2 = k[..., :h].float(), k[..., h:].float()
    return torch.cat([x1 * cos[:T] - x2 * sin[:T], x2 * cos[:T] + x1 * sin[:T]], dim=-1).to(k.dtype)


def _cache_parts(c, s, cache):
    """The caches' contents as lte.h lays them out: keys and values, logits, pool positions and counts, all as views."""
    e, d, rows = DTYPES[c["dtype"]][2], c["d"], c["W"] + c["R"]
    alloc = 256 if c["dtype"] == "bf16" and d == 64 and rows <= 256 else rows
    blocks = cache[256:].view(c["B"] * c["H"], -1)
    a = 2 * alloc * d * e
    b = a + 4 * rows
    return [blocks[:, :a].view(DTYPES[c["dtype"]][0]), blocks[:, a:b].view(torch.float32), blocks[:, b:b + 4 * c["R"] + 8].view(torch.int32)]


def prepare(case, seed):
    c = case
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    B, H, G, T, d, W, R = (c[n] for n in ("B", "H", "G", "T", "d", "W", "R"))
    dt, code, _ = DTYPES[c["dtype"]]
    qk = 1.0 if c["dtype"] == "f32" else d ** -0.25

    def normal(*size, scale=1.0):
        return (torch.randn(size, generator=g, device=dev) * scale).to(dt)

    def shape(n):
        return lte.shape(B, H, n, d, W, R, code, sink=c["sink"], group=G)

    T0 = c["past"] if c["kind"] == "chunk" else T                    # the prompt
    st = {"c": c, "s": shape(T)}
    k, v = normal(B, H, T0, d, scale=qk), normal(B, H, T0, d)
    make = _scorer(c, g, dev)
    conv = make(None)
    if c["half"] and T0 > W:
        z = lte.lte_scores(shape(T0), conv, k, v)[:, :, : T0 - 6]
        sigma = torch.round(z.transpose(0, 1).reshape(H, -1).std(dim=1) * 256) / 256
        conv = make((-sigma * NormalDist().inv_cdf(1.0 - min(0.5, R / (2.0 * (T0 - W))))).to(torch.float32).contiguous())
    st["conv"] = conv
    kr = k
    if c["rope"]:
        angle = torch.arange(1 << 17, device=dev, dtype=torch.float32)[:, None] * 10000.0 ** (-torch.arange(d // 2, device=dev) / (d // 2))
        st["cos"], st["sin"] = angle.cos(), angle.sin()
        kr = _rotated(k, st["cos"], st["sin"])
    if c["kind"] in ("prefill", "train"):
        st.update(k=k, kr=kr, v=v, q=normal(B, H * G, T, d, scale=qk))
        if c["kind"] == "train":
            st.update(dO=normal(B, H * G, T, d), lam=torch.rand((H,), generator=g, device=dev) * 1e-2)
        if c["cache"]:
            st["cache"] = torch.zeros(lte.lte_cache_bytes(st["s"]), dtype=torch.uint8, device=dev)
            st["parts"] = _cache_parts(c, st["s"], st["cache"])
        return st
    # decode, chunk: the cache that the prompt left
    s0 = shape(T0)
    z = lte.lte_scores(s0, conv, k, v)
    idx, cnt = lte.lte_select(s0, z)
    st["cache"] = torch.zeros(lte.lte_cache_bytes(s0), dtype=torch.uint8, device=dev)
    lte.lte_cache_init(s0, conv, kr, v, z, idx, cnt, cache=st["cache"])
    st["parts"] = _cache_parts(c, s0, st["cache"])
    if c["kind"] == "chunk":
        st.update(n=T0, q=normal(B, H * G, T, d, scale=qk), k=normal(B, H, T, d, scale=qk), v=normal(B, H, T, d))
    else:
        n = c["steps"]
        o = torch.empty((n, B, H * G, d), dtype=dt, device=dev)
        lse = torch.empty((n, B, H * G), dtype=torch.float32, device=dev)
        st.update(o=o, lse=lse, tokens=list(zip(normal(n, B, H * G, d, scale=qk), normal(n, B, H, d, scale=qk), normal(n, B, H, d), o, lse)))
    return st


def run(state):
    st = state
    c, s, conv = st["c"], st["s"], st["conv"]
    kind = c["kind"]
    if kind == "decode":
        for q1, k1, v1, o1, lse1 in st["tokens"]:
            lte.lte_attn_decode(s, conv, st["cache"], q1, k1, v1, o1=o1, lse1=lse1)
        if c["rope"]:
            lte.lte_cache_score_unrope(s, conv, st["cache"], st["cos"], st["sin"])
        return [st["o"], st["lse"]] + st["parts"]
    if kind == "chunk":
        o, lse = lte.lte_attn_prefill_chunk(s, conv, st["cache"], st["n"], st["q"], st["k"], st["v"], streaming=c["streaming"])
        st["n"] += c["T"]
        return [o, lse] + st["parts"]
    z = lte.lte_scores(s, conv, st["k"], st["v"])
    idx, cnt = lte.lte_select(s, z)
    o, lse = lte.lte_attn_prefill(s, st["q"], st["kr"], st["v"], idx, cnt)
    if kind == "prefill":
        if c["cache"]:
            lte.lte_cache_init(s, conv, st["kr"], st["v"], z, idx, cnt, cache=st["cache"])
            return [z, idx, cnt, o, lse] + st["parts"]
        return [z, idx, cnt, o, lse]
    count, penalty = lte.lte_sparsity_stats(s, z, st["lam"])
    dq, dk, dv, dw, db = lte.lte_attn_bwd(s, conv, st["q"], st["k"], st["v"], o, lse, st["dO"], z, idx, cnt, lam=st["lam"])
    return [z, idx, cnt, o, lse, count, penalty, dq, dk, dv, dw, db]


def _retained(c, n):
    """Expected retained entries per head after n tokens: half of them pass the threshold, or the half-used budget."""
    out = max(0, n - c["W"])
    return min(c["R"], (min(c["R"] / 2, out / 2) if c["half"] else out / 2) + min(c["sink"], out))


def _pairs(c, past, n):
    """Expected query-key pairs of one head's n queries after `past` tokens: the window, and the retained entries older than it."""
    W, end = c["W"], past + n
    full = max(0, end - max(past, W))                                # queries with a full window
    short = n - full
    window = full * W + short * (past + 1 + past + short) / 2
    cnt, out = _retained(c, end), max(0, end - W)
    seen = (out * out - max(0, past - W) ** 2) / 2 / out * cnt if out else 0.0
    return window + seen


def work(case):
    """Every input read once, every output written once; multiply-adds of the scorer and of the attention's products."""
    c = case
    e = DTYPES[c["dtype"]][2]
    B, H, G, T, d, W, R = (c[n] for n in ("B", "H", "G", "T", "d", "W", "R"))
    heads = B * H
    macs = c["K"] * 2 * d if c["scorer"] == "cnn" else 3 * (2 * d * d + d * d // 2 + d * d // 8) + d // 4
    params = 4 * H * (macs + 1)
    row = 2 * d * e                                                  # a key and a value
    if c["kind"] == "decode":
        # every step reads the block's rows and the pool's logits, moves the popped row and writes the new one; a popped row enters rarely
        per = min(W, T) + _retained(c, T)
        step = heads * (per * row + 4 * R + row + G * (2 * d * e + 4)) + (params if c["scorer"] == "cnn" else 0)
        b, f = c["steps"] * step, c["steps"] * heads * (4.0 * d * G * per + (2 * macs if c["scorer"] == "cnn" else 0))
        if c["rope"]:
            b, f = b + heads * W * (row + 4) + params, f + 2.0 * macs * heads * W
        return {"bytes": b, "flops": f}
    attn = 4.0 * d * G * _pairs(c, c["past"], T)
    if c["kind"] == "chunk":
        state = (min(W, c["past"]) + _retained(c, c["past"])) * row + 8 * (W + R)
        after = (W + _retained(c, c["past"] + T)) * row + 8 * (W + R)
        return {"bytes": heads * (T * (row + G * (2 * d * e + 4)) + state + after) + params, "flops": heads * (attn + 2.0 * macs * T)}
    b = heads * (T * (row + 4 + G * (2 * d * e + 4)) + 4 * (R + 1)) + params
    f = heads * (attn + 2.0 * macs * T)
    if c["rope"]:
        b += heads * T * d * e                                       # the rotated keys beside the others
    if c["cache"]:
        b += heads * ((min(W, T) + _retained(c, T)) * row + 8 * (W + R))
    if c["kind"] == "train":
        # backward: dO read, dq, dk, dv and the scorer's gradients written; what the forward wrote need not be read again in principle
        b += heads * T * (row + G * 2 * d * e) + params
        f += heads * (2.5 * attn + 4.0 * macs * T)
    return {"bytes": b, "flops": f}


def tolerance(case):
    """bf16: rounding of inputs to the products and of results.  fp32: order of summation.  A token whose logit lies within rounding
    of the rank R or of the threshold may be kept or not, which shifts a head's list."""
    if case["dtype"] == "f32":
        return {"rel": 2e-5, "max": 1e-3, "differ": 0.01}
    return {"rel": 1e-2, "max": 0.5, "differ": 0.01}
