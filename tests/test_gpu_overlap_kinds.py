"""Chains that cross the kinds of calls: prefill, decode, wide decode, FP8 decode, latent decode and the small
kernels behind one another on one stream, each call's query the output of the one ahead, with tensor
memory of 512 and of 256 columns, with early signals and without, and with empty sequences between.
Without synchronization, and captured in a graph, they give bit for bit what they give with a
synchronization after every call.
"""
from __future__ import annotations

import pytest
import torch

import paper_2606_21848_gb300 as kl
from tests import _gpu
from tests._gpu import to_dev
from tests._inputs import tiny, tiny_prefill

pytestmark = pytest.mark.gpu
ROUNDS = 4


@pytest.fixture(scope="module", autouse=True)
def lib():
    kl.build()
    kl.load()


# (sequences, heads, value heads, tokens): several CTAs per SM and few; groups of 4 and 16
@pytest.mark.parametrize("B, Hq, Hkv, L", [(4, 32, 8, 1500), (40, 32, 8, 400), (4, 64, 4, 900)])
@pytest.mark.parametrize("order", [0, 1])
def test_chain_of_kinds(B, Hq, Hkv, L, order):
    D, P = 128, 16
    lens = tuple(max(1, L - 37 * i) for i in range(B))
    x = tiny_prefill(B=B, Hq=Hq, Hkv=Hkv, D=D, P=P, lens=lens, q_lens=(1,) * B, seed=270)
    g = to_dev(x)
    dev = _gpu.dev()
    gen = torch.Generator().manual_seed(271)
    w_post = (torch.randn(Hq, D, D, generator=gen) * D ** -0.5).to(torch.bfloat16).to(dev)
    v_new = torch.randn(B, Hkv, D, generator=gen).to(torch.bfloat16).to(dev)
    pages, width = x["v_cache"].shape[0], x["block_table"].shape[1]
    sh = kl.make_shape(B, Hq, Hkv, D, P, pages, width)
    zs = kl.make_latent_shape(B, Hq, Hkv, D, D, P, pages, width)
    latent = Hq // Hkv <= 8
    ws = torch.zeros(max(256, kl.kl_decode_workspace_size(sh, 3), kl.kl_decode_workspace_size(sh, 0),
                         kl.kl_latent_workspace_size(zs, 3) if latent else 0), dtype=torch.uint8, device=dev)
    err = torch.zeros(1, dtype=torch.int32, device=dev)
    codes = torch.empty(g["v_cache"].shape, dtype=torch.uint8, device=dev)
    scales = torch.empty(g["v_cache"].shape[:-1], dtype=torch.float32, device=dev)
    bt, sl, pos, cache, w_r = g["block_table"], g["seq_lens"], g["positions"], g["v_cache"], g["w_r"]
    none = torch.zeros_like(sl)
    cu = g["cu_q"]

    def prefill(q, out):
        kl.kl_append_v_chunk(sh, v_new, bt, sl, cu, B, 1, cache, err)
        kl.kl_prefill_attention(sh, q, w_r, cache, bt, sl, cu, B, 1, out, kl.KL_BF16, err)

    def step(q, out):
        kl.kl_append_v(sh, v_new, bt, pos, cache, err)
        kl.kl_decode_step(sh, q, w_r, v_new, pos, cache, bt, sl, kl.decode_options(3), out, kl.KL_BF16, ws, err)

    def plain(q, out):
        kl.kl_decode_attention(sh, q, w_r, cache, bt, sl, 0, out, kl.KL_BF16, ws, err)

    def fp8(q, out):
        kl.kl_append_v_fp8(sh, v_new, bt, pos, codes, scales, err)
        kl.kl_decode_step_fp8(sh, q, w_r, v_new, pos, codes, scales, bt, sl, 3, out, kl.KL_BF16, ws, err)

    def lat(q, out):
        kl.kl_latent_decode_step(zs, q, w_r, w_post, v_new, pos, cache, bt, sl, 3, out, kl.KL_BF16, ws, err)

    def empty(q, out):
        if latent:
            kl.kl_latent_decode(zs, q, w_r, w_post, cache, bt, none, 1, out, kl.KL_BF16, ws, err)
        kl.kl_decode_attention(sh, q, w_r, cache, bt, none, 1, out, kl.KL_BF16, ws, err)
        plain(q, out)

    kinds = [prefill, step, fp8, plain, empty] + ([lat] if latent else [])
    if order:
        kinds = kinds[::-1] + kinds
    calls = kinds * ROUNDS
    bufs = [torch.empty_like(g["q"]) for _ in range(len(calls) + 1)]

    def run(sync):
        bufs[0].copy_(g["q"])
        for f, q, out in zip(calls, bufs, bufs[1:]):
            f(q, out)
            if sync:
                torch.cuda.synchronize()

    kl.kl_append_v(sh, v_new, bt, pos, cache, err)         # every run starts from the same cache
    kl.kl_quantize_cache_fp8(sh, cache, codes, scales)
    run(True)
    want = [b.clone() for b in bufs[1:]]
    state = [cache.clone(), codes.clone(), scales.clone()]
    for b in bufs:
        b.fill_(float("nan"))
    run(False)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    for i, (a, b) in enumerate(zip(bufs[1:], want)):
        assert torch.isfinite(b).all(), i
        assert torch.equal(a.view(torch.int16), b.view(torch.int16)), f"{i} {calls[i].__name__}"

    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        run(False)
    for b in bufs:
        b.fill_(float("nan"))
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    for i, (a, b) in enumerate(zip(bufs[1:], want)):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16)), f"graph {i} {calls[i].__name__}"
    for a, b in zip((cache, codes, scales), state):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


@pytest.mark.parametrize("Hq, Hkv, splits", [(32, 8, 1), (32, 8, 3), (64, 4, 1), (64, 4, 4)])
def test_copies_and_other_streams_between(Hq, Hkv, splits):
    """Between the calls a copy, a memset or another stream's kernel behind an event: what stands ahead
    of a call in its stream is not a kernel, or more than one thing, and still comes first."""
    B, D, P, L, steps = 6, 128, 16, 1100, 16
    dev = _gpu.dev()
    x = tiny(B=B, Hq=Hq, Hkv=Hkv, D=D, P=P, lens=(L, 40, 700, 1, 300, L), seed=280)
    g = to_dev(x)
    sh = kl.make_shape(B, Hq, Hkv, D, P, x["v_cache"].shape[0], x["block_table"].shape[1])
    ws = torch.zeros(max(256, kl.kl_decode_workspace_size(sh, splits)), dtype=torch.uint8, device=dev)
    err = torch.zeros(1, dtype=torch.int32, device=dev)
    q = [torch.empty_like(g["q"]) for _ in range(steps + 1)]
    out = [torch.empty_like(g["q"]) for _ in range(steps)]
    side = torch.cuda.Stream()
    v_new = g["v_new"]

    def run(sync):
        q[0].copy_(g["q"])
        main = torch.cuda.current_stream()
        for i in range(steps):
            kl.kl_append_v(sh, v_new, g["block_table"], g["positions"], g["v_cache"], err)
            kl.kl_decode_attention(sh, q[i], g["w_r"], g["v_cache"], g["block_table"], g["seq_lens"], splits,
                                   out[i], kl.KL_BF16, ws, err)
            if i % 3 == 0:                              # a copy of the result, on the same stream
                q[i + 1].copy_(out[i])
            elif i % 3 == 1:                            # another stream makes the next query
                side.wait_stream(main)
                with torch.cuda.stream(side):
                    q[i + 1].copy_(out[i]).mul_(1.5)
                main.wait_stream(side)
            else:                                       # a memset, then a kernel
                q[i + 1].zero_()
                q[i + 1].add_(out[i])
            if sync:
                torch.cuda.synchronize()

    run(True)
    want = [b.clone() for b in out]
    for b in out + q:
        b.fill_(float("nan"))
    run(False)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    for i, (a, b) in enumerate(zip(out, want)):
        assert torch.isfinite(b).all() and torch.equal(a.view(torch.int16), b.view(torch.int16)), i
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        run(False)
    for b in out + q:
        b.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    for i, (a, b) in enumerate(zip(out, want)):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16)), f"graph {i}"
