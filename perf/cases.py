"""The work a program using this library has it do, as cases that can be timed and compared.

Each case is one call sequence through the C ABI's Python binding, on inputs that a serving
program holds before the call: cache pool, block table, lengths, projection weights, the new
token's (or chunk's) rows, a zeroed workspace and the output buffer. Four paths:

- ``decode``   ``kl_decode_step``: append the current token and attend over the cache (bf16 rows);
- ``fp8``      ``kl_decode_step_fp8``: the same over E4M3 codes with one fp32 scale per row;
- ``latent``   ``kl_latent_decode_step``: the same over a latent value-only cache;
- ``prefill``  ``kl_append_v_chunk`` then ``kl_prefill_attention``: a chunk of new tokens.

Sizes are the package's own workloads (``paper_2606_21848_gb300/workloads.py``); ``draw`` spreads
over the ranges around them: 1 to 256 sequences, 64 to 131072 cached tokens, pages of 16 to 128
rows, MHA / MQA / GQA with groups of 1 to 32 heads, head dims 64 and 128, equal and ragged
lengths, every split count the library picks or a caller asks for, both forms of W^R and the
composed query, bf16 and (bf16 cache) fp32 outputs.
"""
import math

import torch

from paper_2606_21848_gb300 import _lib

# Numbers of a case: sequences, query and value (latent) heads, head dim, page size, cached tokens
# (len_lo .. len_hi, the current token included), split count (0: the library chooses), W^R ("kv":
# one per value head, "q": one per query head, "none": the query is already composed), output type,
# prefill chunk rows per sequence, and the fraction of cached values scaled by 20.
_DEFAULTS = dict(page=16, splits=0, wr="kv", out="bf16", q_len=0, outliers=0.0)


def _case(name, kind, seqs, q_heads, kv_heads, head_dim, len_lo, len_hi, **more):
    c = dict(_DEFAULTS, kind=kind, seqs=seqs, q_heads=q_heads, kv_heads=kv_heads,
             head_dim=head_dim, len_lo=len_lo, len_hi=len_hi)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one short sequence of a small model: all launch and latency
        _case("tiny_mha", "decode", 1, 4, 4, 64, 256, 256),
        # interactive serving: a few sequences of an 8-value-head GQA model
        _case("small_gqa", "decode", 8, 32, 8, 128, 4096, 4096),
        # one long document; the cache is cut into splits that are merged
        _case("long_context", "decode", 1, 32, 8, 128, 131072, 131072),
        # a serving batch of mixed lengths from one shuffled pool, with outlier values
        _case("ragged_serving", "decode", 64, 32, 8, 128, 512, 32768, outliers=0.01),
        # a full batch of a 70B-class GQA model: the benchmark's default workload
        _case("high_concurrency_70b", "decode", 256, 64, 8, 128, 8192, 8192, page=32),
        # large groups: 16 query heads per value head
        _case("gqa_group16", "decode", 64, 128, 8, 128, 8192, 8192, page=32),
        # multi-query attention: all 32 heads read one value head
        _case("mqa_group32", "decode", 256, 32, 1, 128, 8192, 8192),
        # head dim 64, one value head per query head (GPT-2 style heads)
        _case("mha_d64", "decode", 32, 16, 16, 64, 8192, 8192),
        # the full batch again over the FP8 cache
        _case("fp8_70b", "fp8", 256, 64, 8, 128, 8192, 8192, page=32),
        # latent value-only cache: 4 latent groups of 8 heads
        _case("latent_serving", "latent", 64, 32, 4, 128, 8192, 8192),
        # chunked prefill in serving: 512 new tokens on 7680 cached ones
        _case("prefill_chunked_gqa", "prefill", 8, 32, 8, 128, 8192, 8192, q_len=512),
        # a whole 32K-token prompt, W^R per query head (Qwen2-1.5B's attention)
        _case("prefill_qwen2_32k", "prefill", 1, 12, 2, 128, 32768, 32768, wr="q", q_len=32768),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 5 + ["fp8"] * 2 + ["prefill"] * 2 + ["latent"])
    page = rng.choice([16, 16, 32, 64, 128])
    out, wr, splits, q_len = "bf16", rng.choice(["kv", "kv", "none"]), 0, 0
    seqs = _log(rng, 1, 256)
    if kind == "decode":
        hq, hkv, d = rng.choice([(32, 8, 128), (64, 8, 128), (12, 2, 128), (28, 4, 128), (32, 1, 128),
                                 (128, 8, 128), (8, 8, 128), (16, 16, 64), (12, 12, 64), (32, 8, 64)])
        wr = rng.choice(["kv", "kv", "q", "none"])
        out = rng.choice(["bf16", "bf16", "bf16", "fp32"])
        splits = rng.choice([0, 0, 0, rng.randint(1, 64)])
    elif kind == "fp8":
        hq, hkv, d = rng.choice([(32, 8, 128), (64, 8, 128), (12, 2, 128), (32, 1, 128), (8, 8, 128)])
    elif kind == "latent":
        hq, hkv, d = rng.choice([(32, 4, 128), (16, 4, 128), (32, 8, 128), (8, 1, 128)])
        wr = rng.choice(["kv", "q"])
    else:
        hq, hkv, d = rng.choice([(32, 8, 128), (12, 2, 128), (64, 8, 128), (16, 16, 128)])
        wr = rng.choice(["kv", "q"])
        seqs = _log(rng, 1, 16)
    longest = _log(rng, 64, 131072)
    if kind == "prefill":
        # at most about 1e12 useful FLOPs: a third of the largest listed prompt
        q_len = _log(rng, 1, 8192)
        longest = max(q_len, min(longest, int(1e12 / (4.0 * d * hq * seqs * q_len))))
        if 4.0 * d * hq * seqs * q_len * longest > 1e12:
            q_len = longest = int(math.sqrt(1e12 / (4.0 * d * hq * seqs)))
    # at most 2 GiB of cached rows, counted once per block of 8 query heads that reads them
    row = hkv * d * 2 * max(1, -(-(hq // hkv) // 8))
    longest = max(16, min(longest, (2 << 30) // (row * seqs)))
    q_len = min(q_len, longest)
    shortest = longest if rng.random() < 0.5 else rng.randint(1, longest)
    return _case(None, kind, seqs, hq, hkv, d, shortest, longest, page=page, splits=splits, wr=wr,
                 out=out, q_len=q_len, outliers=rng.choice([0.0, 0.0, 0.01]))


def _lengths(c):
    """Evenly spread lengths len_lo .. len_hi, in order (their sum does not depend on the seed)."""
    n, lo, hi = c["seqs"], c["len_lo"], c["len_hi"]
    return [hi if n == 1 else lo + (hi - lo) * i // (n - 1) for i in range(n)]


def _randn(shape, g, std=1.0):
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)
    return x if std == 1.0 else x * std


def _inputs(c, seed):
    """The tensors of a case (as stored in the cache, before any call)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, Hq, Hkv, D, P = c["seqs"], c["q_heads"], c["kv_heads"], c["head_dim"], c["page"]
    lens = torch.tensor(_lengths(c), dtype=torch.int32)
    lens = lens[torch.randperm(B, generator=torch.Generator().manual_seed(seed))]
    need = [-(-int(n) // P) for n in lens.tolist()]
    pages = sum(need)
    v = _randn((pages, Hkv, P, D), g)
    if c["outliers"]:
        v = torch.where(torch.rand(v.shape, generator=g, device="cuda", dtype=torch.float32)
                        < c["outliers"], v * 20, v)
    perm = torch.randperm(pages, generator=g, device="cuda").to(torch.int32)
    width = -(-c["len_hi"] // P)
    need_t = torch.tensor(need, device="cuda")
    col = torch.arange(width, device="cuda")
    start = torch.cumsum(need_t, 0) - need_t
    at = (start[:, None] + col[None, :]).clamp_max(pages - 1)
    table = torch.where(col[None, :] < need_t[:, None], perm[at], -1).to(torch.int32)
    q_lens = [min(c["q_len"], int(n)) for n in lens.tolist()]
    rows = sum(q_lens) if c["kind"] == "prefill" else B
    s = dict(v=v, table=table.contiguous(), lens=lens.cuda(), pages=pages, width=width,
             positions=(lens - 1).cuda(), q=_randn((rows, Hq, D), g), v_new=_randn((rows, Hkv, D), g),
             w_r=None)
    if c["wr"] != "none":
        s["w_r"] = _randn((Hq if c["wr"] == "q" else Hkv, D, D), g, D ** -0.5)
    if c["kind"] == "latent":
        s["w_post"] = _randn((Hq, D, D), g, D ** -0.5)
    if c["kind"] == "prefill":
        cu = [0]
        for n in q_lens:
            cu.append(cu[-1] + n)
        s["cu"] = torch.tensor(cu, dtype=torch.int32, device="cuda")
        s["rows"], s["max_q"] = rows, max(q_lens)
    return s


def _quantize(v):
    """E4M3 codes and fp32 row scales of bf16 rows: scale = amax / 448, codes of v / scale."""
    codes = torch.empty(v.shape, dtype=torch.uint8, device=v.device)
    scales = torch.empty(v.shape[:-1], dtype=torch.float32, device=v.device)
    n = max(1, (1 << 26) // v[0].numel())
    for i in range(0, v.shape[0], n):
        x = v[i:i + n].float()
        sc = x.abs().amax(-1) / 448.0
        y = x / torch.where(sc > 0, sc, torch.ones_like(sc))[..., None]
        codes[i:i + n] = y.clamp(-448.0, 448.0).to(torch.float8_e4m3fn).view(torch.uint8)
        scales[i:i + n] = sc
    return codes, scales


def prepare(case, seed):
    c = case
    s = _inputs(c, seed)
    B, Hq, Hkv, D = c["seqs"], c["q_heads"], c["kv_heads"], c["head_dim"]
    s["kind"] = c["kind"]
    per_q = c["wr"] == "q"
    if c["kind"] == "latent":
        s["shape"] = _lib.make_latent_shape(B, Hq, Hkv, D, D, c["page"], s["pages"], s["width"], per_q)
        ws = _lib.kl_latent_workspace_size(s["shape"], c["splits"])
    else:
        s["shape"] = _lib.make_shape(B, Hq, Hkv, D, c["page"], s["pages"], s["width"], per_q)
        ws = 0 if c["kind"] == "prefill" else _lib.kl_decode_workspace_size(s["shape"], c["splits"])
    if c["kind"] == "fp8":
        s["codes"], s["scales"] = _quantize(s.pop("v"))
    s["splits"] = c["splits"]
    s["opts"] = _lib.decode_options(c["splits"])
    s["ws"] = torch.zeros(max(256, ws), dtype=torch.uint8, device="cuda")
    s["dtype"] = _lib.KL_FP32 if c["out"] == "fp32" else _lib.KL_BF16
    s["out"] = torch.zeros(s["q"].shape, device="cuda",
                           dtype=torch.float32 if c["out"] == "fp32" else torch.bfloat16)
    s["err"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    return s


def run(state):
    """One decode step or one prefill chunk: the outputs, the updated cache (as the bit patterns
    it stores) and the device error word."""
    s = state
    if s["kind"] == "decode":
        _lib.kl_decode_step(s["shape"], s["q"], s["w_r"], s["v_new"], s["positions"], s["v"],
                            s["table"], s["lens"], s["opts"], s["out"], s["dtype"], s["ws"], s["err"])
    elif s["kind"] == "fp8":
        _lib.kl_decode_step_fp8(s["shape"], s["q"], s["w_r"], s["v_new"], s["positions"], s["codes"],
                                s["scales"], s["table"], s["lens"], s["splits"], s["out"],
                                s["dtype"], s["ws"], s["err"])
        return s["out"], s["codes"], s["scales"].view(torch.int32), s["err"]
    elif s["kind"] == "latent":
        _lib.kl_latent_decode_step(s["shape"], s["q"], s["w_r"], s["w_post"], s["v_new"],
                                   s["positions"], s["v"], s["table"], s["lens"], s["splits"],
                                   s["out"], s["dtype"], s["ws"], s["err"])
    else:
        _lib.kl_append_v_chunk(s["shape"], s["v_new"], s["table"], s["lens"], s["cu"], s["rows"],
                               s["max_q"], s["v"], s["err"])
        _lib.kl_prefill_attention(s["shape"], s["q"], s["w_r"], s["v"], s["table"], s["lens"],
                                  s["cu"], s["rows"], s["max_q"], s["out"], s["dtype"], s["err"])
    return s["out"], s["v"].view(torch.int16), s["err"]


def work(case):
    c = case
    B, Hq, Hkv, D = c["seqs"], c["q_heads"], c["kv_heads"], c["head_dim"]
    lens = _lengths(c)
    tokens = sum(lens)
    row = D + 4 if c["kind"] == "fp8" else 2 * D
    rows = sum(min(c["q_len"], n) for n in lens) if c["kind"] == "prefill" else B
    hw = {"q": Hq, "kv": Hkv, "none": 0}[c["wr"]]
    out_b = 4 if c["out"] == "fp32" else 2
    nbytes = (tokens * Hkv * row                              # cached rows, read once
              + hw * D * D * 2 + rows * Hq * D * (2 + out_b)  # W^R, q, out
              + rows * Hkv * (2 * D + row)                    # the new rows, read and written
              + sum(-(-n // c["page"]) for n in lens) * 4 + 8 * B)
    flops = (2.0 * rows * Hq * D * D if hw else 0.0)
    if c["kind"] == "prefill":
        # row i of a chunk of n rows sees L - n + i + 1 tokens
        for L in lens:
            n = min(c["q_len"], L)
            flops += 4.0 * Hq * D * (n * (L - n) + n * (n + 1) / 2)
    else:
        flops += 4.0 * tokens * Hq * D
    if c["kind"] == "latent":
        nbytes += Hq * D * D * 2
        flops += 4.0 * rows * Hq * D * D
    return {"bytes": float(nbytes), "flops": flops}


def _rows_of(c, s, b, n):
    """Sequence b's n cached rows in order, [Hkv][n][D] in 64 bits, without the new ones."""
    ids = s["table"][b, :-(-n // c["page"])].long()
    if c["kind"] == "fp8":
        x = (s["codes"][ids].view(torch.float8_e4m3fn).float().double()
             * s["scales"][ids].double()[..., None])
    else:
        x = s["v"][ids].double()
    return x.transpose(0, 1).reshape(c["kv_heads"], -1, c["head_dim"])[:, :n].clone()


def exact(case, seed):
    """The outputs in 64 bits from the definition: q_r = q W^R, one softmax over the rows that the
    query sees, the weighted sum of the same rows. (None in the place of the cache: it is copied.)"""
    c = case
    s = _inputs(c, seed)
    B, Hq, Hkv, D = c["seqs"], c["q_heads"], c["kv_heads"], c["head_dim"]
    G = Hq // Hkv
    scale = D ** -0.5
    v_new = s["v_new"].double()
    if c["kind"] == "fp8":
        s["codes"], s["scales"] = _quantize(s.pop("v"))
        codes, scales = _quantize(s["v_new"])
        v_new = codes.view(torch.float8_e4m3fn).float().double() * scales.double()[..., None]
    q = s["q"].double()
    if s["w_r"] is not None:
        w = s["w_r"].double()
        w = w if c["wr"] == "q" else w.repeat_interleave(G, 0)
        q = torch.einsum("rhk,hkj->rhj", q, w)
    if c["kind"] == "latent":
        q = torch.einsum("rhj,hkj->rhk", q, s["w_post"].double())
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    cu = s["cu"].tolist() if c["kind"] == "prefill" else list(range(B + 1))
    for b, L in enumerate(s["lens"].tolist()):
        x = _rows_of(c, s, b, L)
        n = cu[b + 1] - cu[b]
        if n == 0:
            continue
        x[:, L - n:] = v_new[cu[b]:cu[b + 1]].transpose(0, 1)
        qb = q[cu[b]:cu[b + 1]].reshape(n, Hkv, G, D).permute(1, 2, 0, 3)   # [Hkv][G][n][D]
        step = max(1, (1 << 28) // (Hq * L)) if n > 1 else 1
        for i in range(0, n, step):
            j = min(n, i + step)
            seen = L - n + j
            p = torch.matmul(qb[:, :, i:j].reshape(Hkv, -1, D), x[:, :seen].transpose(1, 2))
            p = p.view(Hkv, G, j - i, seen).mul_(scale)
            if n > 1:
                pos = torch.arange(L - n + i, L - n + j, device="cuda")
                p.masked_fill_(torch.arange(seen, device="cuda")[None, :] > pos[:, None], -math.inf)
            p = torch.softmax(p, -1).view(Hkv, -1, seen)
            o = torch.matmul(p, x[:, :seen]).view(Hkv, G, j - i, D)
            out[cu[b] + i:cu[b] + j] = o.permute(2, 0, 1, 3).reshape(j - i, Hq, D)
    if c["kind"] == "latent":
        out = torch.einsum("rhk,hkd->rhd", out, s["w_post"].double())
    return (out, None, None, None) if c["kind"] == "fp8" else (out, None, None)
