"""Performance cases of the attention and GEMM library: what a serving or training program
has it do, through the Python entry points.

A case is a dict of plain values.  ``kind`` names the entry point:

* ``prefill``  loom_attn_fwd on dense [B, H, S, D] tensors
* ``varlen``   loom_attn_fwd_varlen on a ragged batch of packed tokens
* ``decode``   loom_attn_decode on a contiguous cache (o, lse and workspace kept by the caller)
* ``paged``    loom_attn_decode_paged on a paged cache (o, lse and workspace kept by the caller)
* ``gemm``     loom_gemm_bf16, C = A B, or with ``bt`` C = A W^T (a linear layer's weight)

Sequence lengths of a batch are a fixed set for a case (evenly spaced from ``lo`` to
``hi``), so that its work does not depend on the seed; the seed deals them to the
sequences and makes every tensor's values.
"""
import math
import random

import torch

import paper_2609_29219_gb300 as loom

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def _prefill(B, Hq, Hkv, Sq, Skv, D, causal, lse=False):
    return {"kind": "prefill", "B": B, "Hq": Hq, "Hkv": Hkv, "Sq": Sq, "Skv": Skv, "D": D, "causal": causal, "lse": lse}


def _varlen(B, Hq, Hkv, lo, hi, D, causal, lse=False):
    return {"kind": "varlen", "B": B, "Hq": Hq, "Hkv": Hkv, "lo": lo, "hi": hi, "D": D, "causal": causal, "lse": lse}


def _decode(B, Hq, Hkv, cap, lo, hi, D, splits=0):
    return {"kind": "decode", "B": B, "Hq": Hq, "Hkv": Hkv, "cap": cap, "lo": lo, "hi": hi, "D": D, "splits": splits}


def _paged(B, Hq, Hkv, page, lo, hi, D, layout, splits=0):
    return {"kind": "paged", "B": B, "Hq": Hq, "Hkv": Hkv, "page": page, "lo": lo, "hi": hi, "D": D, "layout": layout,
            "splits": splits}


def _gemm(M, N, K, bt):
    return {"kind": "gemm", "M": M, "N": N, "K": K, "bt": bt}


def listed():
    named = [
        # the smallest call: two heads, one query tile, where the launch is what costs
        ("prefill_tiny", _prefill(1, 2, 2, 128, 128, 64, False)),
        # a batch of bidirectional (encoder) sequences: the benchmark's headline
        ("prefill_b4_s2048", _prefill(4, 32, 32, 2048, 2048, 128, False)),
        # the same batch in a decoder: training forward or a batch of prompts
        ("prefill_b4_s2048_causal", _prefill(4, 32, 32, 2048, 2048, 128, True)),
        # one chunk of a prompt against the keys before it (chunked prefill; odd sizes)
        ("prefill_chunk_515_of_3001", _prefill(1, 32, 8, 515, 3001, 128, True, lse=True)),
        # one long prompt of a model with 64-wide heads
        ("prefill_s8192_d64_causal", _prefill(1, 64, 16, 8192, 8192, 64, True)),
        # a server's batch of prompts of all lengths, packed; the largest call
        ("varlen_16_seqs", _varlen(16, 32, 8, 1024, 8192, 128, True, lse=True)),
        # one user, early in a conversation: the latency of one decode step
        ("decode_one_short", _decode(1, 32, 8, 2048, 1000, 1000, 128)),
        # a decode step of a busy server, split count fixed by the caller
        ("decode_b16_8k", _decode(16, 32, 8, 8192, 4096, 8192, 128, splits=16)),
        # one user with a very long context
        ("decode_one_131072", _decode(1, 32, 8, 131072, 131072, 131072, 128)),
        # the busy server with a paged cache of small pages
        ("paged_b16_8k_page16", _paged(16, 32, 8, 16, 4096, 8192, 128, "nhd")),
        # the QKV projection of a decode step: few rows, a weight that is read once
        ("linear_m16_n6144_k4096", _gemm(16, 6144, 4096, True)),
        # the benchmark's square product: a projection over a long batch of tokens
        ("gemm_8192", _gemm(8192, 8192, 8192, False)),
    ]
    return [dict(c, name=n) for n, c in named]


MOST_FLOPS = 3.0e12  # a drawn case's most (the largest listed case has more)
MOST_BYTES = 5.0e8   # and the most bytes of a cache or an operand set


def _log(rng, lo, hi):
    """A whole number from lo to hi, spread over the logarithm."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


HEADS = ((32, 32), (32, 8), (64, 16), (16, 16), (16, 2), (8, 1), (8, 8), (6, 3))


def _draw_once(rng):
    kind = rng.choice(("prefill", "prefill", "varlen", "decode", "decode", "paged", "gemm", "gemm"))
    D = rng.choice((64, 128, 128))
    Hq, Hkv = rng.choice(HEADS)
    if kind == "prefill":
        Sq = _log(rng, 64, 8192)
        causal = rng.random() < 0.6
        Skv = Sq if rng.random() < 0.6 else _log(rng, Sq, 16384)
        return _prefill(_log(rng, 1, 16), Hq, Hkv, Sq, Skv, D, causal, rng.random() < 0.4)
    if kind == "varlen":
        hi = _log(rng, 256, 8192)
        return _varlen(_log(rng, 2, 32), Hq, Hkv, _log(rng, max(1, hi // 16), hi), hi, D, rng.random() < 0.8, rng.random() < 0.4)
    if kind == "decode":
        hi = _log(rng, 128, 131072)
        lo = hi if rng.random() < 0.3 else _log(rng, max(1, hi // 16), hi)
        cap = hi if rng.random() < 0.5 else min(131072, hi + hi // 4)
        return _decode(_log(rng, 1, 64), Hq, Hkv, cap, lo, hi, D, rng.choice((0, 0, 0, 4, 16)))
    if kind == "paged":
        hi = _log(rng, 128, 32768)
        lo = _log(rng, max(1, hi // 16), hi)
        return _paged(_log(rng, 1, 64), Hq, Hkv, rng.choice((16, 16, 32, 64, 128)), lo, hi, D, rng.choice(("nhd", "nhd", "hnd")),
                      rng.choice((0, 0, 0, 16)))
    # a linear layer or a product: few rows to many, widths a multiple of 8
    return _gemm(_log(rng, 1, 16384), 8 * _log(rng, 32, 2048), 8 * _log(rng, 32, 2048), rng.random() < 0.6)


def draw(rng: random.Random):
    while True:
        c = _draw_once(rng)
        w = work(c)
        held = c["B"] * c["cap"] * c["Hkv"] * c["D"] * 4 if c["kind"] == "decode" else w["bytes"]
        if w["flops"] <= MOST_FLOPS and held <= MOST_BYTES:
            return c


# ------------------------------------------------------------------ work
def _lengths(case):
    B, lo, hi = case["B"], case["lo"], case["hi"]
    return [hi] if B == 1 else [lo + round((hi - lo) * i / (B - 1)) for i in range(B)]


def _pairs(sq, skv, causal):
    return sq * skv - (sq * (sq - 1) // 2 if causal else 0)


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2 * (M * K + K * N + M * N), "flops": 2 * M * N * K}
    B, Hq, Hkv, D = case["B"], case["Hq"], case["Hkv"], case["D"]
    if kind == "prefill":
        sq, skv = case["Sq"], case["Skv"]
        pairs, rows, keys = B * _pairs(sq, skv, case["causal"]), B * sq, B * skv
    elif kind == "varlen":
        ls = _lengths(case)
        pairs, rows, keys = sum(_pairs(n, n, case["causal"]) for n in ls), sum(ls), sum(ls)
    else:
        pairs = keys = sum(_lengths(case))
        rows = B
    b = 4 * rows * Hq * D + 4 * keys * Hkv * D
    if kind in ("decode", "paged") or case["lse"]:
        b += 4 * rows * Hq
    return {"bytes": b, "flops": 4 * D * Hq * pairs}


# ------------------------------------------------------------------ inputs
def _normal(gen, shape, std=1.0):
    t = torch.randn(shape, generator=gen, device=DEV, dtype=torch.bfloat16)
    return t if std == 1.0 else t.mul_(std)


def _dealt(case, seed):
    """The case's sequence lengths in the order that the seed deals them."""
    ls = _lengths(case)
    random.Random(seed).shuffle(ls)
    return ls


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    kind, s = case["kind"], {"case": case}
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        s["a"] = _normal(gen, (M, K))
        s["b"] = _normal(gen, (N, K) if case["bt"] else (K, N), K ** -0.5)
        return s
    B, Hq, Hkv, D = case["B"], case["Hq"], case["Hkv"], case["D"]
    if kind == "prefill":
        s["q"] = _normal(gen, (B, Hq, case["Sq"], D))
        s["k"] = _normal(gen, (B, Hkv, case["Skv"], D))
        s["v"] = _normal(gen, (B, Hkv, case["Skv"], D))
        return s
    ls = _dealt(case, seed)
    if kind == "varlen":
        offs = [0]
        for n in ls:
            offs.append(offs[-1] + n)
        s["q"] = _normal(gen, (offs[-1], Hq, D))
        s["k"] = _normal(gen, (offs[-1], Hkv, D))
        s["v"] = _normal(gen, (offs[-1], Hkv, D))
        s["cu"] = torch.tensor(offs, dtype=torch.int32, device=DEV)
        s["max_seqlen"] = max(ls)
        return s
    s["q"] = _normal(gen, (B, Hq, 1, D))
    s["lens"] = torch.tensor(ls, dtype=torch.int32, device=DEV)
    s["o"] = torch.empty_like(s["q"])
    s["lse"] = torch.empty((B, Hq), dtype=torch.float32, device=DEV)
    if kind == "decode":
        cap = case["cap"]
        shape = (B, Hkv, cap, D)
    else:
        page = case["page"]
        max_pages = -(-max(ls) // page)
        used = [-(-n // page) for n in ls]
        pages = sum(used) + 8  # a pool with a few free pages
        order = torch.randperm(pages, generator=gen, device=DEV).to(torch.int32).cpu()
        table = torch.zeros((B, max_pages), dtype=torch.int32)
        at = 0
        for b, n in enumerate(used):
            table[b, :n] = order[at:at + n]
            at += n
        s["table"] = table.to(DEV)
        cap = max_pages * page
        shape = (pages, page, Hkv, D) if case["layout"] == "nhd" else (pages, Hkv, page, D)
    s["k"] = _normal(gen, shape)
    s["v"] = _normal(gen, shape)
    need = loom.loom_attn_decode_workspace_bytes(B, Hq, Hkv, cap, D, case["splits"])
    s["workspace"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    return s


# ------------------------------------------------------------------ one pass
def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "prefill":
        return loom.loom_attn_fwd(state["q"], state["k"], state["v"], causal=c["causal"], return_lse=c["lse"])
    if kind == "varlen":
        return loom.loom_attn_fwd_varlen(state["q"], state["k"], state["v"], state["cu"], state["cu"], state["max_seqlen"],
                                         causal=c["causal"], return_lse=c["lse"])
    if kind == "decode":
        return loom.loom_attn_decode(state["q"], state["k"], state["v"], state["lens"], state["o"], state["lse"],
                                     state["workspace"], num_splits=c["splits"])
    if kind == "paged":
        return loom.loom_attn_decode_paged(state["q"], state["k"], state["v"], state["table"], state["lens"], state["o"],
                                           state["lse"], state["workspace"], num_splits=c["splits"], layout=c["layout"])
    return loom.loom_gemm_bf16(state["a"], state["b"], b_transposed=c["bt"])


# ------------------------------------------------------------------ the same in 64 bits
def _attend(q, k, v, causal):
    """q [g, sq, D] against one kv head's k, v [skv, D], all float64: (o, lse)."""
    g, sq, D = q.shape
    skv = k.shape[0]
    o = torch.empty_like(q)
    lse = torch.empty((g, sq), dtype=torch.float64, device=q.device)
    step = max(1, min(sq, (1 << 26) // (g * skv)))
    for r in range(0, sq, step):
        e = min(sq, r + step)
        n = min(skv, e + skv - sq) if causal else skv
        s = (q[:, r:e].reshape(-1, D) @ k[:n].T).view(g, e - r, n).mul_(D ** -0.5)
        if causal:
            i = torch.arange(r, e, device=q.device)[:, None] + (skv - sq)
            s.masked_fill_(torch.arange(n, device=q.device)[None, :] > i, -math.inf)
        m = s.amax(-1, keepdim=True)
        s.sub_(m).exp_()
        total = s.sum(-1, keepdim=True)
        lse[:, r:e] = (m + total.log())[..., 0]
        o[:, r:e] = (s.view(-1, n) @ v[:n]).view(g, e - r, D) / total
    return o, lse


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "gemm":
        b = s["b"].double()
        return s["a"].double() @ (b.T if case["bt"] else b)
    Hq, Hkv = case["Hq"], case["Hkv"]
    g = Hq // Hkv
    o = torch.empty(s["q"].shape, dtype=torch.float64, device=DEV)
    q, k, v = s["q"], s["k"], s["v"]
    if kind == "prefill":
        lse = torch.empty(q.shape[:3], dtype=torch.float64, device=DEV)
        for b in range(case["B"]):
            for h in range(Hkv):
                hs = slice(h * g, (h + 1) * g)
                o[b, hs], lse[b, hs] = _attend(q[b, hs].double(), k[b, h].double(), v[b, h].double(), case["causal"])
        return (o, lse) if case["lse"] else o
    if kind == "varlen":
        lse = torch.empty((Hq, q.shape[0]), dtype=torch.float64, device=DEV)
        offs = s["cu"].tolist()
        for a, e in zip(offs, offs[1:]):
            for h in range(Hkv):
                hs = slice(h * g, (h + 1) * g)
                x, y = _attend(q[a:e, hs].transpose(0, 1).double().contiguous(), k[a:e, h].double(), v[a:e, h].double(),
                               case["causal"])
                o[a:e, hs], lse[hs, a:e] = x.transpose(0, 1), y
        return (o, lse) if case["lse"] else o
    lse = torch.empty((case["B"], Hq), dtype=torch.float64, device=DEV)
    for b, n in enumerate(s["lens"].tolist()):
        if kind == "paged":
            pages = s["table"][b, : -(-n // case["page"])].long()
            kb, vb = k[pages], v[pages]
            if case["layout"] == "hnd":
                kb, vb = kb.transpose(1, 2), vb.transpose(1, 2)
            kb, vb = (x.reshape(-1, Hkv, case["D"])[:n].transpose(0, 1) for x in (kb, vb))
        else:
            kb, vb = k[b, :, :n], v[b, :, :n]
        for h in range(Hkv):
            hs = slice(h * g, (h + 1) * g)
            x, y = _attend(q[b, hs].double(), kb[h].double(), vb[h].double(), False)
            o[b, hs], lse[b, hs] = x, y[:, 0]
    return o, lse


def tolerance(case):
    # About four times what was measured against exact().  GEMM: one rounding of the result
    # to bf16 (rel 1.7e-3, max 3.9e-3).  Attention: that, and the rounding of the
    # probabilities to bf16 before they meet V (rel 2.1e-3 to 2.4e-3; max 1.1e-2 where all
    # rows see many keys, up to 5.0e-2 where the first causal rows see few and are large).
    if case["kind"] == "gemm":
        return {"rel": 0.0066, "max": 0.016}
    return {"rel": 0.0094, "max": 0.2 if case.get("causal") else 0.06}
