"""Rows whose weights are far apart (1 % outlier values x20) move their reference several times. The fp32
output is then no further off from 64 bits than a prefill that walks whole 128-token tiles and moves
a warp's references when one row's tile maximum passes its own by 2^8: that one is replayed here in
64 bits but for the rounding of the weights to fp16.

Bound: both round every weight once, so the rms errors differ by what each leaves exact (a weight of
exactly 1) and by chance, which between seeds is 1 % to 2 %; 2 % is allowed. With half tiles and the
same 2^8 the error was 6 % larger.
"""
from __future__ import annotations

import math

import pytest
import torch

from tests import _gpu
from tests._gpu import to_dev
from tests._inputs import tiny_prefill
from tests.test_gpu_prefill import lib, run_prefill  # noqa: F401 (lib: fixture)

pytestmark = pytest.mark.gpu


def _replay(q, v, L, n):
    """(exact, replayed) outputs of n <= 32 rows of one head: q [n][D], v [L][D], in 64 bits."""
    s = q @ v.T / math.sqrt(q.shape[1]) / math.log(2)
    s.masked_fill_(torch.arange(L, device=s.device) > torch.arange(L - n, L, device=s.device)[:, None], -math.inf)
    exact = torch.softmax(s * math.log(2), -1) @ v
    m = torch.full((n,), -math.inf, dtype=torch.float64, device=s.device)
    o, l = torch.zeros_like(exact), torch.zeros_like(m)
    for t in range(0, L, 128):
        new = torch.maximum(m, s[:, t:t + 128].amax(-1))
        if bool((new > m + 8).any()):
            f = torch.where(m == -math.inf, torch.zeros_like(m), torch.exp2(m - new))
            o, l, m = o * f[:, None], l * f, new
        p = torch.exp2(s[:, t:t + 128] - m[:, None])
        o, l = o + p.half().double() @ v[t:t + 128], l + p.sum(-1)
    return exact, o / l[:, None]


def test_outlier_rows():
    B, Hq, Hkv, D, n = 6, 32, 8, 128, 32
    lens = (500, 800, 1100, 1400, 1700, 2000)
    x = tiny_prefill(B=B, Hq=Hq, Hkv=Hkv, D=D, P=16, lens=lens, q_lens=(n,) * B, seed=180,
                     wr_per_query_head=True)
    g = torch.Generator().manual_seed(181)
    big = torch.rand(x["v_cache"].shape, generator=g) < 0.01
    x["v_cache"] = torch.where(big, x["v_cache"] * 20, x["v_cache"])
    got, err = run_prefill(x)
    assert err == 0
    d = to_dev(x)
    q = torch.einsum("thk,hkj->thj", d["q"].double(), d["w_r"].double())
    mine = ref = 0.0
    for b, L in enumerate(lens):
        v = d["v_cache"][d["block_table"][b, :-(-L // 16)].long()].double().transpose(0, 1).reshape(Hkv, -1, D)[:, :L]
        for h in range(Hq):
            exact, replayed = _replay(q[b * n:(b + 1) * n, h], v[h // (Hq // Hkv)], L, n)
            ref += float((replayed - exact).square().sum())
            mine += float((got[b * n:(b + 1) * n, h].double() - exact).square().sum())
    assert math.sqrt(mine) <= 1.02 * math.sqrt(ref), math.sqrt(mine / ref)
