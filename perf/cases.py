"""The attention calls whose speed is watched: what a serving program has this library do.

A case is one call of a public entry point on tensors that are already in device memory.  There
are four kinds: ``prefill`` (``fa_forward`` on a dense batch), ``varlen`` (a packed batch of
requests of different lengths, with its keys packed as well or in pages), ``decode`` (16-bit
cache, contiguous or in pages, one or several new tokens per sequence) and ``decode_fp8`` (FP8
e4m3 cache).  ``listed()`` names twelve of them, ``draw()`` makes more of the same ranges.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2410_16663_b200 import binding as fa

DEV = "cuda"
DTYPES = {"fp16": torch.float16, "bf16": torch.bfloat16}
# factors of the FP8 cache: N(0,1) keys and values lie well inside e4m3's range at these
K_SCALE, V_SCALE = 0.25, 0.125


def listed():
    return [
        # one short prompt on two heads, the smallest configuration: launch and latency
        dict(name="prefill_short", kind="prefill", B=1, Hq=2, Hkv=2, Sq=512, Skv=512, d=128, dtype="fp16", causal=True),
        # eight prompts of 512 tokens, 7B-class heads: the usual batch of short prompts
        dict(name="prefill_prompts", kind="prefill", B=8, Hq=32, Hkv=32, Sq=512, Skv=512, d=128, dtype="fp16", causal=True),
        # one prompt on the five heads that one GPU of eight holds: few heads, a few thousand keys
        dict(name="prefill_5heads", kind="prefill", B=1, Hq=5, Hkv=5, Sq=4096, Skv=4096, d=128, dtype="fp16", causal=True),
        # the benchmark's prefill
        dict(name="prefill_2k", kind="prefill", B=4, Hq=32, Hkv=32, Sq=2048, Skv=2048, d=128, dtype="fp16", causal=True),
        # one long prompt: the largest case
        dict(name="prefill_32k", kind="prefill", B=1, Hq=32, Hkv=32, Sq=32768, Skv=32768, d=128, dtype="bf16", causal=True),
        # the last chunk of a chunked prefill with grouped heads, sizes that are multiples of nothing
        dict(name="prefill_chunk", kind="prefill", B=2, Hq=64, Hkv=8, Sq=1001, Skv=7951, d=128, dtype="bf16", causal=True),
        # a serving engine's packed batch of whole prompts
        dict(name="varlen_serving", kind="varlen", n=32, Hq=32, Hkv=32, len_lo=256, len_hi=8192, lens=31, page=0, chunk=0,
             d=128, dtype="bf16"),
        # image batch of a vision transformer: 197 tokens, head dimension 64, no mask
        dict(name="vision", kind="prefill", B=1024, Hq=12, Hkv=12, Sq=197, Skv=197, d=64, dtype="fp16", causal=False),
        # a full decode batch with grouped heads, the benchmark's lengths
        dict(name="decode_batch", kind="decode", B=64, Sq=1, Hq=32, Hkv=8, len_lo=1024, len_hi=32768, lens=1021, page=0,
             d=128, dtype="fp16"),
        # one sequence on one GPU's five heads: the latency of a single user's next token
        dict(name="decode_one", kind="decode", B=1, Sq=1, Hq=5, Hkv=5, len_lo=8192, len_hi=8192, lens=1, page=0, d=128,
             dtype="fp16"),
        # a chat batch on a paged cache with the small pages that serving engines default to
        dict(name="decode_paged", kind="decode", B=48, Sq=1, Hq=32, Hkv=8, len_lo=100, len_hi=8000, lens=5, page=16, d=128,
             dtype="bf16"),
        # the 8-bit cache in pages, bf16 model
        dict(name="decode_fp8", kind="decode_fp8", B=64, Sq=1, Hq=32, Hkv=8, len_lo=1024, len_hi=32768, lens=9, page=64,
             d=128, dtype="bf16"),
    ]


def _log_int(rng, lo, hi):
    """An integer in [lo, hi], even over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


_MOST_FLOPS = 4 * 32 * 128 * 32768 * 32769 / 2      # the long prompt's
_MOST_BYTES = 12e9                                  # about the time of the long prompt's arithmetic


def draw(rng):
    while True:
        case = _draw(rng)
        w = work(case)
        if w["flops"] <= 0.9 * _MOST_FLOPS and w["bytes"] <= _MOST_BYTES:
            return case


def _draw(rng):
    kind = rng.choice(["prefill", "prefill", "chunk", "varlen", "vision", "decode", "decode", "decode_fp8"])
    dtype = rng.choice(["fp16", "bf16"])
    hq, hkv = rng.choice([(32, 32), (32, 8), (64, 8), (8, 8), (5, 5)])
    if kind == "prefill":
        s = _log_int(rng, 128, 32768)
        most = max(1, min(16, 65536 // s))
        return dict(kind="prefill", B=_log_int(rng, 1, most), Hq=hq, Hkv=hkv, Sq=s, Skv=s, d=128, dtype=dtype,
                    causal=rng.random() < 0.8)
    if kind == "chunk":
        skv = _log_int(rng, 1024, 32768)
        return dict(kind="prefill", B=_log_int(rng, 1, 4), Hq=hq, Hkv=hkv, Sq=_log_int(rng, 128, min(2048, skv)), Skv=skv,
                    d=128, dtype=dtype, causal=True)
    if kind == "varlen":
        hi = _log_int(rng, 512, 8192)
        page = rng.choice([0, 0, 128, 256])
        return dict(kind="varlen", n=_log_int(rng, 2, 32), Hq=hq, Hkv=hkv, len_lo=max(1, hi // 32), len_hi=hi,
                    lens=rng.randrange(1 << 20), page=page, chunk=512 if page and rng.random() < 0.5 else 0, d=128, dtype=dtype)
    if kind == "vision":
        s = rng.choice([197, 197, rng.randint(144, 256)])
        h = rng.choice([3, 6, 12, 16])
        return dict(kind="prefill", B=_log_int(rng, 32, 1024), Hq=h, Hkv=h, Sq=s, Skv=s, d=64, dtype=dtype, causal=False)
    hi = _log_int(rng, 512, 32768)
    b = _log_int(rng, 1, 64)
    page = rng.choice([0, 16, 64, 256])
    sq = rng.choice([1, 1, 1, 2, 4]) if kind == "decode" else 1
    return dict(kind=kind, B=b, Sq=sq, Hq=hq, Hkv=hkv, len_lo=max(8, hi // 32), len_hi=hi, lens=rng.randrange(1 << 20),
                page=page, d=128, dtype=dtype)


def _lens(case):
    """The case's sequence lengths (key counts); part of the case, not of its inputs' values."""
    rng = random.Random(case["lens"])
    n = case["n"] if case["kind"] == "varlen" else case["B"]
    return [rng.randint(case["len_lo"], case["len_hi"]) for _ in range(n)]


def _chunks(case, lens):
    """Query rows of each request of a packed batch: the whole prompt, or its last chunk."""
    return [min(x, case["chunk"]) if case["chunk"] else x for x in lens]


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _normal(shape, dtype, gen):
    return torch.empty(shape, dtype=dtype, device=DEV).normal_(generator=gen)


def _normal_fp8(shape, scale, gen):
    """N(0,1) divided by its factor and rounded to e4m3, as bit patterns, a slab at a time."""
    out = torch.empty(shape, dtype=torch.uint8, device=DEV)
    flat = out.view(-1)
    step = 1 << 28
    for i in range(0, flat.numel(), step):
        part = flat[i:i + step]
        x = torch.empty(part.numel(), dtype=torch.bfloat16, device=DEV).normal_(0.0, 1.0 / scale, generator=gen)
        part.copy_(x.to(torch.float8_e4m3fn).view(torch.uint8))
    return out


def _table(lens, page, seed):
    """Block table of sequences whose pages were handed out in a random order; -1 past a sequence's end."""
    need = [-(-x // page) for x in lens]
    pages = sum(need)
    order = list(range(pages))
    random.Random(seed).shuffle(order)
    table = torch.full((len(lens), max(need)), -1, dtype=torch.int32)
    at = 0
    for b, n in enumerate(need):
        table[b, :n] = torch.tensor(order[at:at + n], dtype=torch.int32)
        at += n
    return table.to(DEV), pages


def prepare(case, seed):
    gen = _gen(seed)
    d, hq, hkv, dt = case["d"], case["Hq"], case["Hkv"], DTYPES[case["dtype"]]
    st = {"case": case, "scale": 1.0 / math.sqrt(d)}
    if case["kind"] == "prefill":
        B, sq, skv = case["B"], case["Sq"], case["Skv"]
        st["q"] = _normal((B, sq, hq, d), dt, gen)
        st["k"] = _normal((B, skv, hkv, d), dt, gen)
        st["v"] = _normal((B, skv, hkv, d), dt, gen)
        st["o"] = torch.empty_like(st["q"])
        st["lse"] = torch.empty(B, hq, sq, dtype=torch.float32, device=DEV)
        return st
    lens = _lens(case)
    if case["kind"] == "varlen":
        rows = _chunks(case, lens)
        st["q"] = _normal((sum(rows), hq, d), dt, gen)
        st["o"] = torch.empty_like(st["q"])
        st["lse"] = torch.empty(hq, sum(rows), dtype=torch.float32, device=DEV)
        st["cu_q"] = torch.tensor([0] + rows).cumsum(0).to(torch.int32).to(DEV)
        st["max_q"], st["max_k"] = max(rows), max(lens)
        if case["page"]:
            st["table"], pages = _table(lens, case["page"], seed)
            st["seqlens"] = torch.tensor(lens, dtype=torch.int32, device=DEV)
            shape = (pages, case["page"], hkv, d)
        else:
            st["cu_k"] = torch.tensor([0] + lens).cumsum(0).to(torch.int32).to(DEV)
            shape = (sum(lens), hkv, d)
        st["k"], st["v"] = _normal(shape, dt, gen), _normal(shape, dt, gen)
        return st
    # decode: the query rows are the last positions of the cache
    B, sq = case["B"], case["Sq"]
    st["q"] = _normal((B, sq, hq, d), dt, gen)
    st["o"] = torch.empty_like(st["q"])
    st["lse"] = torch.empty(B, hq, sq, dtype=torch.float32, device=DEV)
    st["seqlens"] = torch.tensor(lens, dtype=torch.int32, device=DEV)
    if case["page"]:
        st["table"], pages = _table(lens, case["page"], seed)
        shape, most = (pages, case["page"], hkv, d), st["table"].shape[1] * case["page"]
    else:
        st["table"], most = None, max(lens)
        shape = (B, most, hkv, d)
    if case["kind"] == "decode_fp8":
        st["k"], st["v"] = _normal_fp8(shape, K_SCALE, gen), _normal_fp8(shape, V_SCALE, gen)
    else:
        st["k"], st["v"] = _normal(shape, dt, gen), _normal(shape, dt, gen)
    need = fa.fa_decode_append_workspace_bytes(B, sq, hq, hkv, most, d)
    st["ws"] = torch.empty(max(16, need), dtype=torch.uint8, device=DEV)
    return st


def run(st):
    case = st["case"]
    q, k, v, o, lse, scale = st["q"], st["k"], st["v"], st["o"], st["lse"], st["scale"]
    if case["kind"] == "prefill":
        fa.fa_forward(q, k, v, o, lse, case["causal"], scale)
    elif case["kind"] == "varlen":
        if case["page"]:
            fa.fa_forward_varlen_paged(q, k, v, st["table"], o, lse, st["cu_q"], st["seqlens"], st["max_q"], st["max_k"], True,
                                       scale)
        else:
            fa.fa_forward_varlen(q, k, v, o, lse, st["cu_q"], st["cu_k"], st["max_q"], st["max_k"], True, scale)
    elif case["kind"] == "decode":
        fa.fa_decode_ex(q, k, v, o, lse, st["seqlens"], scale, st["ws"], block_table=st["table"])
    elif case["page"]:
        call = fa.fa_decode_fp8_paged_bf16 if case["dtype"] == "bf16" else fa.fa_decode_fp8_paged
        call(q, k, v, st["table"], o, lse, st["seqlens"], scale, K_SCALE, V_SCALE, st["ws"])
    else:
        call = fa.fa_decode_fp8_bf16 if case["dtype"] == "bf16" else fa.fa_decode_fp8
        call(q, k, v, o, lse, st["seqlens"], scale, K_SCALE, V_SCALE, st["ws"])
    return {"o": o, "lse": lse}


def work(case):
    """q, the keys and values of every sequence and the outputs once; 4*d operations for each visible
    (query, key) pair of each query head."""
    d, hq, hkv = case["d"], case["Hq"], case["Hkv"]
    if case["kind"] == "prefill":
        sets = [(case["Sq"], case["Skv"])] * case["B"]
        causal = case["causal"]
    else:
        lens = _lens(case)
        causal = True
        sets = list(zip(_chunks(case, lens), lens)) if case["kind"] == "varlen" else [(case["Sq"], x) for x in lens]
    rows, keys, pairs = 0, 0, 0
    for nq, nk in sets:
        rows += nq
        keys += nk
        pairs += nq * (nk - nq) + nq * (nq + 1) // 2 if causal else nq * nk
    kv_bytes = 1 if case["kind"] == "decode_fp8" else 2
    return {"bytes": rows * hq * (2 * d * 2 + 4) + 2 * keys * hkv * d * kv_bytes, "flops": 4 * d * hq * pairs}


def tolerance(case):
    # Four times what the calls differ from the same arithmetic in 64 bits: 2.8e-4 with fp16 (the rounding of the stored
    # output and of the probabilities), 2.4e-3 with bf16; the largest single difference over the output's root mean square
    # is 3.8e-3 (fp16) and 5.4e-2 (bf16, the first rows of a causal prompt, whose values are several times the rms).
    if case["dtype"] == "fp16":
        return {"rel": 1.1e-3, "max": 1.5e-2}
    return {"rel": 9e-3, "max": 0.2 if case["kind"] in ("prefill", "varlen") else 4e-2}
