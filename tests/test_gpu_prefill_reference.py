"""The reference of a prefill row's weights covers its first 128 tokens: where the row's largest weight
lies there, it is exactly 1 and takes no part in the weights' rounding to fp16.

Each row has one token that outweighs every other by 2^3 to 2^7.5 (below the 2^8 that move a
reference later on) and holds nearly all of the output, so the output's error is that weight's.
Bound: the routed query's pair of bf16 operands leaves a score, at most 8, an error of about
8 * 2^-17, which moves a weight p of the normalized sum by p (1 - p) ln 2 of that, at most 1.1e-5 of
the token's values; the other tokens' rounded weights add less than 2^-11 of their values, 1/50 of
it, 1e-5. Together 2.1e-5 at most, and rms below 1e-5. A rounded largest weight leaves
p 2^-11 / sqrt(12) to twice that, rms 5e-5 or more.
"""
from __future__ import annotations

import math

import pytest
import torch

from tests._inputs import tiny_prefill
from tests.test_gpu_prefill import lib, run_prefill  # noqa: F401 (lib: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at", [5, 63, 64, 100, 127])
def test_largest_weight_of_the_first_tokens_is_exact(at):
    B, H, D, L = 16, 8, 128, 128
    x = tiny_prefill(B=B, Hq=H, Hkv=H, D=D, P=16, lens=(L,) * B, q_lens=(1,) * B, seed=170, table="identity")
    g = torch.Generator().manual_seed(171)
    x["w_r"] = torch.eye(D).expand(H, D, D).contiguous().to(torch.bfloat16)
    q = x["q"].double()                                             # [B][H][D]
    v = torch.randn(B, L, H, D, generator=g) * 0.02
    # log2 of the token's weight over the others': 3 .. 7.5, different in every row
    lead = 3.0 + 4.5 * torch.rand(B, H, 1, generator=g)
    v[:, at] = lead * math.log(2) * math.sqrt(D) * (q / q.square().sum(-1, keepdim=True)).float()
    x["v_cache"] = v.view(B, 8, 16, H, D).transpose(2, 3).reshape(B * 8, H, 16, D).to(torch.bfloat16).contiguous()
    got, err = run_prefill(x)
    assert err == 0
    v = v.to(torch.bfloat16).double()
    p = torch.softmax(torch.einsum("bhd,blhd->bhl", q, v) / math.sqrt(D), -1)
    want = torch.einsum("bhl,blhd->bhd", p, v)
    size = v[:, at].abs()
    rel = (got.cpu().double() - want).norm(dim=-1) / size.norm(dim=-1)
    assert float(rel.square().mean().sqrt()) <= 1e-5, float(rel.square().mean().sqrt())
