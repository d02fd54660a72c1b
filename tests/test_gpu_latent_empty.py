"""Latent decode steps whose sequences are all empty, between steps that hold tokens, on one workspace
and without synchronization: the empty step's absorbed queries are stored while nothing else of its
call runs, and must still be ordered ahead of the next call's in the same place. Each step must
give bit for bit what the same chain gives with a synchronization after every call.
"""
from __future__ import annotations

import pytest
import torch

import paper_2606_21848_gb300 as kl
from tests import _gpu
from tests._gpu import to_dev
from tests._inputs import tiny

pytestmark = pytest.mark.gpu
STEPS = 12


@pytest.fixture(scope="module", autouse=True)
def lib():
    kl.build()
    kl.load()


# one block of query rows and two (more than 128 sequences); merged inside the decode and direct
@pytest.mark.parametrize("B, splits", [(3, 1), (3, 4), (150, 1)])
@pytest.mark.parametrize("empty", ["zero", "out of range"])
def test_empty_steps_between(B, splits, empty):
    Hq, Hl, D = 16, 4, 128
    x = tiny(B=B, Hq=Hq, Hkv=Hl, D=D, P=16, lens=((1500, 700, 129) * 50)[:B], seed=31)
    g = to_dev(x)
    gen = torch.Generator().manual_seed(5)
    w_post = (torch.randn(Hq, D, D, generator=gen) * D ** -0.5).to(torch.bfloat16).to(_gpu.dev())
    sh = kl.make_latent_shape(B, Hq, Hl, D, D, 16, x["v_cache"].shape[0], x["block_table"].shape[1])
    ws = torch.zeros(kl.kl_latent_workspace_size(sh, splits), dtype=torch.uint8, device=_gpu.dev())
    err = torch.zeros(1, dtype=torch.int32, device=_gpu.dev())
    none = torch.full_like(g["seq_lens"], 0 if empty == "zero" else -1)
    bufs = [torch.empty_like(g["q"]) for _ in range(STEPS + 1)]

    def run(sync):
        bufs[0].copy_(g["q"])
        for i in range(STEPS):
            # empty, empty, then a step whose query is the last output that is not zero
            held = i % 3 == 2
            src = bufs[i - 2] if held else g["q"]
            kl.kl_latent_decode(sh, src, g["w_r"], w_post, g["v_cache"], g["block_table"],
                                g["seq_lens"] if held else none, splits, bufs[i + 1], kl.KL_BF16, ws, err)
            if sync:
                torch.cuda.synchronize()
        return [b.clone() for b in bufs[1:]]

    want = run(True)
    for b in bufs:
        b.fill_(float("nan"))
    got = run(False)
    torch.cuda.synchronize()
    assert int(err.item()) == (0 if empty == "zero" else kl.KL_FLAG_BAD_LENGTH)
    for i, (a, b) in enumerate(zip(got, want)):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16)), f"step {i}"
        assert torch.isfinite(a).all() and bool((a != 0).any()) == (i % 3 == 2), f"step {i}"
