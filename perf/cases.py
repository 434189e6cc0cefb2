"""Workloads of the library's public entry points: cache writes (prefill) and
decode steps over every cache format, from one short sequence to a million
cached tokens.

A case is a dict of plain values:

  kind      "prefill": one cache write of the prompts' tokens;
            "decode":  attention over a cache written beforehand;
            "step":    what a serving loop does per generated token: write each
                       sequence's newest token(s), then attend
  cache     "int4", "int2" (this library's blocks), "c4r4" (the paper's page)
            or "bf16" (the comparison cache)
  protect   sink4/local128 BF16 protection rows written and read
  batch, heads, q_tokens
            sequences, query heads per token, query tokens per sequence
  len_lo, len_hi
            the sequences' lengths, spread over this range (the same for every
            seed); for a prefill the prompts' lengths
  skip      prefill only: tokens of each sequence that earlier calls wrote

Inputs follow the repository's synthetic workloads: latents N(0, 1) with
per-channel gains and outlier channels (Student-t for INT2), RoPE-rotated keys,
queries N(0, 1/512) and N(0, 1/64), a random block table.
"""
from __future__ import annotations

import math

import torch

import paper_2609_36760_gb300 as Q

TAU = 1.0 / math.sqrt(192.0)
BLOCK = 64
TOKEN_BYTES = {"int4": 324, "int2": 196, "c4r4": 320, "bf16": 1152}
CHUNK_TOKENS = 1 << 17  # tokens drawn and written per call while a cache is prepared


def _case(name, kind, cache, batch, heads, lo, hi, protect=False, q_tokens=1, skip=0):
    c = {"kind": kind, "cache": cache, "protect": protect, "batch": batch, "heads": heads, "q_tokens": q_tokens,
         "len_lo": lo, "len_hi": hi, "skip": skip}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # A single short chat turn, 16 heads on this GPU: all latency.
        _case("tiny_b1_h16", "decode", "int4", 1, 16, 256, 256),
        # A lightly loaded server: a few ragged conversations, all 128 heads, protected cache.
        _case("small_b8_h128_protected", "step", "int4", 8, 128, 300, 2500, protect=True),
        # The DeepSeek-V3-shaped serving step, 4096 cached tokens and one appended.
        _case("dsv3_b64_h128_int4", "step", "int4", 64, 128, 4097, 4097),
        # The same step on the paper's serving configuration: its own page with protection.
        _case("dsv3_b64_h128_c4r4_protected", "step", "c4r4", 64, 128, 4097, 4097, protect=True),
        # The same step on the unquantised cache that the method is compared with.
        _case("dsv3_b64_h128_bf16", "step", "bf16", 64, 128, 4097, 4097),
        # Speculative verification: two query tokens per sequence on ragged contexts.
        _case("verify2_b48_h128_int4", "step", "int4", 48, 128, 1500, 6000, q_tokens=2),
        # INT2 content at 32K context, heavy-tailed latents: the largest decode.
        _case("int2_b32_h128_l32k", "decode", "int2", 32, 128, 32768, 32768),
        # Few very long contexts of skewed lengths, heads sharded to 64.
        _case("long_b4_h64_128k", "decode", "int4", 4, 64, 16384, 131072),
        # Cache-pressure serving mix: many sequences, heads sharded to 16.
        _case("serve_b128_h16_mix", "step", "int4", 128, 16, 1024, 16384),
        # Head counts and lengths that fill no tile: INT2 with protection, 100 heads.
        _case("ragged_b33_h100_int2_protected", "step", "int2", 33, 100, 70, 9001, protect=True),
        # Prompt processing: the prompts of several requests written in one call.
        _case("prefill_int4_32k", "prefill", "int4", 8, 1, 2500, 5700),
        # A later chunk of a chunked prefill on the paper's serving configuration.
        _case("prefill_c4r4_protected_6k", "prefill", "c4r4", 3, 1, 1900, 2100, protect=True, skip=4096),
    ]


_MAX_FLOPS = 2.9e11  # the largest listed decode
_MAX_TOKENS = 1_100_000


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    cache = rng.choice(["int4", "int4", "int2", "c4r4", "bf16"])
    protect = cache != "bf16" and rng.random() < 0.4
    if rng.random() < 0.25:
        total = _log_int(rng, 64, 65536)
        batch = rng.randint(1, max(1, min(16, total // 40)))
        mean = max(1, total // batch)
        lo = max(1, int(mean * rng.uniform(0.4, 1.0)))
        return _case(None, "prefill", cache, batch, 1, lo, max(lo, 2 * mean - lo), protect=protect,
                     skip=rng.choice([0, 0, rng.randint(1, 9000)]))
    heads = rng.choice([16, 20, 32, 64, 100, 128, 128])
    q_tokens = rng.choice([1, 1, 1, 2, 4]) if cache in ("int4", "int2") else 1
    batch = _log_int(rng, 1, 128)
    hi = _log_int(rng, 65, 131072)
    room = min(_MAX_TOKENS, int(_MAX_FLOPS / (2 * 1088 * heads * q_tokens)))
    if cache == "bf16":
        room //= 2
    hi = max(9, min(hi, room // batch))
    lo = max(9, int(hi * rng.uniform(0.1, 1.0)))
    return _case(None, rng.choice(["decode", "step"]), cache, batch, heads, min(lo, hi), hi, protect=protect,
                 q_tokens=q_tokens)


# ---------------------------------------------------------------- inputs
def _lengths(case):
    """The sequences' lengths: len_lo .. len_hi, both ends taken, in a scattered order."""
    B, lo, hi = case["batch"], case["len_lo"], case["len_hi"]
    if B == 1:
        return [hi]
    return [lo + ((i * (hi - lo)) // (B - 1)) for i in sorted(range(B), key=lambda i: (i * 0.6180339887) % 1.0)]


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1_000_003 + stream)
    return g


def _gains(case, seed):
    g = _gen(seed, 1)
    gain = torch.exp(0.5 * torch.randn(512, generator=g, device="cuda"))
    if case["cache"] != "int2":
        gain[torch.randperm(512, generator=g, device="cuda")[:4]] *= 8.0
    return gain


def _tokens(case, seed):
    """Yields (sequence ids, positions, latent bf16 [n, 512], k_pe bf16 [n, 64])
    over all tokens of all sequences, sequence by sequence, in pieces."""
    gain, g = _gains(case, seed), _gen(seed, 2)
    skip = case["skip"]
    lens = torch.tensor(_lengths(case), device="cuda")
    sid = torch.repeat_interleave(torch.arange(case["batch"], device="cuda"), lens)
    first = torch.cumsum(lens, 0) - lens
    pos = torch.arange(sid.numel(), device="cuda") - first[sid] + skip
    freq = 10000.0 ** (-torch.arange(32, device="cuda", dtype=torch.float64) / 32.0)
    for a in range(0, sid.numel(), CHUNK_TOKENS):
        s, p = sid[a:a + CHUNK_TOKENS], pos[a:a + CHUNK_TOKENS]
        n = s.numel()
        x = torch.randn(n, 512, generator=g, device="cuda")
        if case["cache"] == "int2":  # Student-t with 4 degrees of freedom
            u = 1.0 - torch.rand(2, n, 512, generator=g, device="cuda")
            x = x / torch.sqrt(-0.5 * (torch.log(u[0]) + torch.log(u[1]))).clamp_min(1e-3)
        k = torch.randn(n, 64, generator=g, device="cuda")
        ang = p.double()[:, None] * freq[None, :]
        c, d = torch.cos(ang).float(), torch.sin(ang).float()
        kr = torch.cat([k[:, :32] * c - k[:, 32:] * d, k[:, :32] * d + k[:, 32:] * c], 1)
        yield s.int(), p.int(), (x * gain).bfloat16(), kr.bfloat16()


def _queries(case, seed):
    g = _gen(seed, 3)
    B, T, H = case["batch"], case["q_tokens"], case["heads"]
    shape = (B, T, H) if T > 1 else (B, H)
    ql = torch.randn(*shape, 512, generator=g, device="cuda") / math.sqrt(512.0)
    qp = torch.randn(*shape, 64, generator=g, device="cuda") / 8.0
    return ql.bfloat16(), qp.bfloat16()


# ---------------------------------------------------------------- the calls
def _append(case, st, seq_ids, positions, latent, k_pe, lens_after):
    if case["cache"] == "bf16":
        Q.bf16_append(st["pool"], latent, k_pe, seq_ids, positions, st["table"], st["err"])
    elif case["cache"] == "c4r4":
        Q.quant_append_c4r4(st["pool"], latent, k_pe, seq_ids, positions, st["table"], st["err"],
                            seq_lens=lens_after if case["protect"] else None, prot=st["prot"])
    elif case["protect"]:
        Q.quant_append_protected(st["pool"], 4 if case["cache"] == "int4" else 2, latent, k_pe, seq_ids, positions,
                                 st["table"], lens_after, st["prot"], st["err"])
    else:
        Q.quant_append(st["pool"], 4 if case["cache"] == "int4" else 2, latent, k_pe, seq_ids, positions,
                       st["table"], st["err"])


def _decode(case, st):
    bits = 2 if case["cache"] == "int2" else 4
    if case["q_tokens"] > 1:
        Q.mla_decode_multi(st["pool"], bits, st["ql"], st["qp"], st["table"], st["lens"], TAU, st["out"], st["lse"],
                           st["ws"], st["err"], prot=st["prot"])
    elif case["cache"] == "bf16":
        Q.mla_decode_bf16cache(st["pool"], st["ql"], st["qp"], st["table"], st["lens"], TAU, st["out"], st["lse"],
                               st["ws"], st["err"])
    elif case["cache"] == "c4r4":
        Q.mla_decode_c4r4(st["pool"], st["ql"], st["qp"], st["table"], st["lens"], TAU, st["out"], st["lse"],
                          st["ws"], st["err"], prot=st["prot"])
    elif case["protect"]:
        Q.mla_decode_protected(st["pool"], bits, st["ql"], st["qp"], st["table"], st["lens"], st["prot"], TAU,
                               st["out"], st["lse"], st["ws"], st["err"])
    else:
        Q.mla_decode(st["pool"], bits, st["ql"], st["qp"], st["table"], st["lens"], TAU, st["out"], st["lse"],
                     st["ws"], st["err"])


def prepare(case, seed):
    """The cache, block table, queries and buffers that a serving program holds."""
    B, T, H = case["batch"], case["q_tokens"], case["heads"]
    lens = _lengths(case)
    ends = [n + case["skip"] for n in lens]
    nblk = [(n + BLOCK - 1) // BLOCK for n in ends]
    total = sum(nblk)
    perm = torch.randperm(total, generator=_gen(seed, 4), device="cuda").int()
    table = torch.full((B, max(nblk)), -1, dtype=torch.int32, device="cuda")
    at = 0
    for b, n in enumerate(nblk):
        table[b, :n] = perm[at:at + n]
        at += n
    bb = {"int4": lambda: Q.block_bytes(4), "int2": lambda: Q.block_bytes(2), "c4r4": Q.c4r4_page_bytes,
          "bf16": Q.bf16_block_bytes}[case["cache"]]()
    st = {"case": case, "table": table, "err": torch.zeros(1, dtype=torch.int32, device="cuda"),
          "pool": torch.zeros((total, bb), dtype=torch.uint8, device="cuda"),
          "prot": torch.zeros((B, 132, 576), dtype=torch.bfloat16, device="cuda") if case["protect"] else None,
          "lens": torch.tensor(ends, dtype=torch.int32, device="cuda")}
    if case["kind"] == "prefill":
        parts = list(_tokens(case, seed))
        st["new"] = [torch.cat([p[i] for p in parts]) for i in range(4)]
        return st
    new = T if case["kind"] == "step" else 0  # tokens of each sequence that run() writes
    before = st["lens"] - new
    late = []
    for s, p, lat, kpe in _tokens(case, seed):
        old = p < before[s.long()]
        if new:
            late.append((s[~old], p[~old], lat[~old], kpe[~old]))
            s, p, lat, kpe = s[old], p[old], lat[old], kpe[old]
        _append(case, st, s, p, lat, kpe, before)
    st["new"] = [torch.cat([x[i] for x in late]) for i in range(4)] if new else None
    st["ql"], st["qp"] = _queries(case, seed)
    st["out"] = torch.zeros(st["ql"].shape, dtype=torch.float32, device="cuda")
    st["lse"] = torch.zeros(st["ql"].shape[:-1], dtype=torch.float32, device="cuda")
    st["ws"] = Q.workspace_for(B, T * H)
    return st


def run(st):
    case = st["case"]
    if st["new"] is not None:
        _append(case, st, *st["new"], st["lens"])
    written = {"pool": st["pool"]} if st["new"] is not None else {}
    if st["new"] is not None and st["prot"] is not None:
        written["prot"] = st["prot"]
    if case["kind"] == "prefill":
        return written
    _decode(case, st)
    return {"out": st["out"], "lse": st["lse"], **written}


def work(case):
    T, H, B, per = case["q_tokens"], case["heads"], case["batch"], TOKEN_BYTES[case["cache"]]
    lens = _lengths(case)
    rows = sum(min(n, 132) for n in lens)  # rows the protection buffer holds
    if case["kind"] == "prefill":
        return {"bytes": sum(lens) * (1152 + per) + (rows * 1152 if case["protect"] else 0), "flops": 0}
    read = sum(lens) * per if not case["protect"] else (sum(lens) - rows) * per + rows * 1152
    new = B * T * (1152 + per + (1152 if case["protect"] else 0)) if case["kind"] == "step" else 0
    return {"bytes": read + new + B * T * H * (1152 + 2048 + 4), "flops": 2 * 1088 * H * T * sum(lens)}


# ---------------------------------------------------------------- 64-bit values
def _quantised(x, bits, paper, content):
    """s (q - z) in 64 bits for rows of 64-channel groups [n, groups, 64] (bf16
    input), with the cache formats' own rounding of the stored scale."""
    m = float(2 ** bits - 1)
    x = x.float()
    lo, hi = x.amin(-1, keepdim=True), x.amax(-1, keepdim=True)
    s = (hi - lo).clamp_min(1e-8) / m
    if paper:
        s = s.bfloat16().float() if content else s
        z = torch.round(-lo / s).clamp(0, m)
        q = torch.round(x / s + z).clamp(0, m)
        return s.double() * (q - z).double()
    s = s.half().float()
    s = torch.where(s == 0, torch.full_like(s, 2.0 ** -24), s).clamp_max(65504.0).double()
    z = torch.round(-lo.double() / s).clamp(0, m)
    return s * (torch.round(x.double() / s + z).clamp(0, m) - z)


def exact(case, seed):
    if case["kind"] == "prefill":
        return None
    B, T, H = case["batch"], case["q_tokens"], case["heads"]
    bits, paper = (2 if case["cache"] == "int2" else 4), case["cache"] == "c4r4"
    lens = _lengths(case)
    end = torch.tensor(lens, device="cuda")
    ql, qp = _queries(case, seed)
    ql, qp = ql.reshape(B, T * H, 512).double(), qp.reshape(B, T * H, 64).double()
    top = torch.full((B, T * H), -math.inf, dtype=torch.float64, device="cuda")
    den = torch.zeros(B, T * H, dtype=torch.float64, device="cuda")
    num = torch.zeros(B, T * H, 512, dtype=torch.float64, device="cuda")
    for s, p, lat, kpe in _tokens(case, seed):
        for b in torch.unique(s).tolist():
            mine = s == b
            pos, x, k = p[mine], lat[mine], kpe[mine]
            c, r = x.double(), k.double()
            if case["cache"] != "bf16":
                cq = _quantised(x.view(-1, 8, 64), bits, paper, True).reshape(-1, 512)
                rq = _quantised(k.view(-1, 1, 64), 4, paper, False).reshape(-1, 64)
                if case["protect"]:
                    kept = ((pos < 4) | (pos >= end[b] - 128))[:, None]
                    cq, rq = torch.where(kept, c, cq), torch.where(kept, r, rq)
                c, r = cq, rq
            sc = TAU * (ql[b] @ c.T + qp[b] @ r.T)
            if T > 1:  # query token t sees positions up to length - T + t
                t = torch.arange(T * H, device="cuda") // H
                sc = sc.masked_fill(pos[None, :] > (end[b] - T + t)[:, None], -math.inf)
            new = torch.maximum(top[b], sc.amax(-1))
            ref = torch.where(torch.isinf(new), torch.zeros_like(new), new)
            w, old = torch.exp(sc - ref[:, None]), torch.exp(top[b] - ref)
            den[b] = den[b] * old + w.sum(-1)
            num[b] = num[b] * old[:, None] + w @ c
            top[b] = new
    shape = (B, T, H) if T > 1 else (B, H)
    out = torch.where(den[..., None] > 0, num / den[..., None].clamp_min(1e-300), torch.zeros_like(num))
    got = {"out": out.reshape(*shape, 512), "lse": (top + torch.log(den)).reshape(shape)}
    if case["kind"] == "step":
        got["pool"] = None
        if case["protect"]:
            got["prot"] = None
    return got
