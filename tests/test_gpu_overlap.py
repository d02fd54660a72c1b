"""Kernels that start under the end of the one ahead of them keep stream order: chains of calls in
which each call's query is the previous call's output (written and read by this library's kernels
back to back, or with a torch kernel between), with no synchronization, must give bit for bit what
the same chain gives with a synchronization after every call -- also when captured in a graph.
"""
from __future__ import annotations

import pytest
import torch

import paper_2606_21848_gb300 as kl
from tests import _gpu
from tests._gpu import to_dev
from tests._inputs import tiny, tiny_prefill

pytestmark = pytest.mark.gpu
STEPS = 10


@pytest.fixture(scope="module", autouse=True)
def lib():
    kl.build()
    kl.load()


def _chain(kind, B, Hq, Hkv, D, L, splits):
    """A function that runs one call (query buffer -> output buffer) on fixed inputs."""
    lens = (L, max(1, L // 3))[:B] + (L // 2,) * max(0, B - 2)
    if kind == "prefill":
        x = tiny_prefill(B=B, Hq=Hq, Hkv=Hkv, D=D, P=16, lens=lens, q_lens=tuple(min(n, 150) for n in lens),
                         seed=7)
    else:
        x = tiny(B=B, Hq=Hq, Hkv=Hkv, D=D, P=16, lens=lens, seed=7)
    g = to_dev(x)
    pages, width = x["v_cache"].shape[0], x["block_table"].shape[1]
    err = torch.zeros(1, dtype=torch.int32, device=_gpu.dev())
    T = x["q"].shape[0]
    gen = torch.Generator().manual_seed(3)
    v_new = torch.randn(T, Hkv, D, generator=gen).to(torch.bfloat16).to(_gpu.dev())
    w_post = (torch.randn(Hq, D, D, generator=gen) * D ** -0.5).to(torch.bfloat16).to(_gpu.dev())
    if kind == "latent":
        sh = kl.make_latent_shape(B, Hq, Hkv, D, D, 16, pages, width)
        ws = torch.zeros(kl.kl_latent_workspace_size(sh, splits), dtype=torch.uint8, device=_gpu.dev())
    else:
        sh = kl.make_shape(B, Hq, Hkv, D, 16, pages, width)
        ws = torch.zeros(max(256, kl.kl_decode_workspace_size(sh, splits)), dtype=torch.uint8,
                         device=_gpu.dev())
    codes = torch.empty(g["v_cache"].shape, dtype=torch.uint8, device=_gpu.dev())
    scales = torch.empty(g["v_cache"].shape[:-1], dtype=torch.float32, device=_gpu.dev())
    if kind == "fp8":
        kl.kl_quantize_cache_fp8(sh, g["v_cache"], codes, scales)
    bt, sl, pos = g["block_table"], g["seq_lens"], g["positions"]

    def call(q, out):
        if kind == "decode":
            kl.kl_append_v(sh, v_new, bt, pos, g["v_cache"], err)
            kl.kl_decode_step(sh, q, g["w_r"], v_new, pos, g["v_cache"], bt, sl,
                              kl.decode_options(splits), out, kl.KL_BF16, ws, err)
        elif kind == "fp8":
            kl.kl_decode_step_fp8(sh, q, g["w_r"], v_new, pos, codes, scales, bt, sl, splits, out,
                                  kl.KL_BF16, ws, err)
        elif kind == "latent":
            kl.kl_latent_decode_step(sh, q, g["w_r"], w_post, v_new, pos, g["v_cache"], bt, sl, splits,
                                     out, kl.KL_BF16, ws, err)
        else:
            kl.kl_append_v_chunk(sh, v_new, bt, sl, g["cu_q"], T, 150, g["v_cache"], err)
            kl.kl_prefill_attention(sh, q, g["w_r"], g["v_cache"], bt, sl, g["cu_q"], T, 150, out,
                                    kl.KL_BF16, err)

    return call, g["q"], err


@pytest.mark.parametrize("kind, B, Hq, Hkv, D, L, splits", [
    ("decode", 2, 8, 8, 128, 400, 1), ("decode", 2, 64, 8, 128, 3000, 4),
    ("decode", 1, 8, 8, 64, 2000, 3), ("decode", 24, 128, 8, 128, 700, 1),
    ("decode", 1, 32, 1, 128, 9000, 20), ("fp8", 2, 32, 8, 128, 3000, 5), ("fp8", 3, 8, 1, 128, 300, 1),
    ("latent", 3, 16, 4, 128, 1500, 0), ("prefill", 2, 8, 2, 128, 700, 0)])
def test_chained_calls(kind, B, Hq, Hkv, D, L, splits):
    call, q0, err = _chain(kind, B, Hq, Hkv, D, L, splits)
    bufs = [torch.empty_like(q0) for _ in range(STEPS + 1)]

    def run(sync, torch_between):
        bufs[0].copy_(q0)
        for i in range(STEPS):
            if torch_between and i:
                bufs[i].mul_(2.0)
            call(bufs[i], bufs[i + 1])
            if sync:
                torch.cuda.synchronize()
        return [b.clone() for b in bufs[1:]]

    for between in (False, True):
        want = run(True, between)
        for b in bufs:
            b.fill_(float("nan"))
        got = run(False, between)
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        for i, (a, b) in enumerate(zip(got, want)):
            assert torch.equal(a.view(torch.int16), b.view(torch.int16)), f"step {i}, between {between}"

    # the same chain captured in a graph and replayed twice
    want = run(True, False)
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        bufs[0].copy_(q0)
        for i in range(STEPS):
            call(bufs[i], bufs[i + 1])
    for b in bufs:
        b.fill_(float("nan"))
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    for i, b in enumerate(want):
        assert torch.equal(bufs[i + 1].view(torch.int16), b.view(torch.int16)), f"graph step {i}"
