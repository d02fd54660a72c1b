"""GPU parity of the prefill's block layouts: several heads of a group in one 128-row block (chunks
that leave it room), and clusters of 2, 4 and 8 CTAs that split a block's cache tiles and merge
their states, with ranks that get no tiles, rows that the query box does not fill and references
that differ between the ranks."""
from __future__ import annotations

import math

import pytest
import torch

import paper_2606_21848_gb300 as kl
from tests._gpu import assert_parity
from tests._inputs import tiny_prefill
from tests.test_gpu_prefill import lib, oracle_prefill, run_prefill  # noqa: F401 (lib: fixture)

pytestmark = pytest.mark.gpu


def _check(x, what, **kw):
    got, err = run_prefill(x, **kw)
    assert err == 0
    assert_parity(got.float().cpu().numpy(), oracle_prefill(x, 1.0 / math.sqrt(128)), what)


# (heads per value head, chunk): blocks of 1 to 32 heads, full and with rows left over
@pytest.mark.parametrize("G, chunk", [(8, 1), (8, 3), (8, 17), (6, 21), (6, 22), (7, 18), (4, 33),
                                      (32, 4), (12, 40), (8, 130), (1, 5)])
@pytest.mark.parametrize("per_q", [False, True])
def test_heads_per_block(G, chunk, per_q):
    lens = (1500, 700, 129)
    x = tiny_prefill(B=3, Hq=2 * G, Hkv=2, D=128, P=16, lens=lens, q_lens=(chunk, max(0, chunk - 1), chunk)
                     if chunk <= 129 else (chunk, chunk - 1, 129), seed=130 + G, wr_per_query_head=per_q)
    _check(x, f"G {G} chunk {chunk} per_q {per_q}")


# one value head: 1, 3, 9, 20, 70 and 100 blocks (clusters of 8, 8, 8, 4, 2 and single CTAs)
@pytest.mark.parametrize("B", [1, 3, 9, 20, 70, 100])
@pytest.mark.parametrize("out", [kl.KL_FP32, kl.KL_BF16])
def test_clusters(B, out):
    lens = tuple((2000, 1, 64, 300, 1025, 128, 900)[i % 7] for i in range(B))
    x = tiny_prefill(B=B, Hq=2, Hkv=1, D=128, P=16, lens=lens, q_lens=tuple(min(n, 60) for n in lens),
                     seed=140 + B)
    _check(x, f"B {B}", out_dtype=out)


def test_cluster_moving_reference():
    """Rows that grow along the sequence: the ranks' references are far apart."""
    x = tiny_prefill(B=1, Hq=4, Hkv=1, D=128, P=16, lens=(1800,), q_lens=(20,), seed=150, table="identity")
    v = x["v_cache"].float().view(113, 1, 16, 128)
    ramp = 0.05 + 6.0 * (torch.arange(113 * 16) / 1800.0) ** 2
    x["v_cache"] = (v * ramp.view(113, 1, 16, 1)).to(torch.bfloat16)
    _check(x, "growing rows")


def test_cluster_range_flag():
    """A value beyond fp16 in one rank's share makes the rows non-finite and raises the flag."""
    x = tiny_prefill(B=1, Hq=4, Hkv=1, D=128, P=16, lens=(1800,), q_lens=(3,), seed=151, table="identity")
    x["v_cache"][40, 0, 3, 7] = 69632.0
    got, err = run_prefill(x)
    assert err == kl.KL_FLAG_RANGE
    assert not torch.isfinite(got[:, :, 7]).any()
