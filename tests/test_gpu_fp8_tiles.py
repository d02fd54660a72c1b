"""GPU parity of the FP8 decode at the edges of its tiles and softmax groups: 0 to 6 tiles with
remainders around the 32-token output steps, groups of 1 to 8 heads that do and do not fill their
blocks of 4, and rows that grow along the sequence, so that the references and the weights' power
of two move while both groups have tiles in flight."""
from __future__ import annotations

import math

import pytest
import torch

import oracle
from paper_2606_21848_gb300.workloads import bf16_bits
from tests._gpu import assert_parity
from tests._inputs import tiny
from tests.test_gpu_fp8 import fp8_cache, lib, run_fp8  # noqa: F401 (lib: fixture)

pytestmark = pytest.mark.gpu

EDGES = (0, 1, 31, 32, 33, 127, 128, 129, 160, 161, 255, 256, 257, 384, 385, 640, 641, 700)


def _want(x, codes, scales):
    return oracle.decode_fp8(bf16_bits(x["q"]), bf16_bits(x["w_r"]), codes, scales,
                             x["block_table"].numpy(), x["seq_lens"].numpy(), scale=1.0 / math.sqrt(128))


@pytest.mark.parametrize("G, P", [(1, 16), (3, 128), (4, 32), (5, 16), (8, 64), (12, 16)])
def test_tile_edges(G, P):
    x = tiny(B=len(EDGES), Hq=2 * G, Hkv=2, D=128, P=P, lens=EDGES, seed=110 + G)
    codes, scales = fp8_cache(x)
    got, err = run_fp8(x, codes, scales, num_splits=1)
    assert err == 0
    assert_parity(got.cpu().numpy(), _want(x, codes, scales), f"G {G}")


@pytest.mark.parametrize("G, splits", [(4, 1), (8, 1), (8, 2)])
def test_moving_reference_and_scale(G, splits):
    x = tiny(B=2, Hq=2 * G, Hkv=2, D=128, P=16, lens=(1100, 1100), seed=120, table="identity")
    v = x["v_cache"].float().view(2, 69, 2, 16, 128)      # [b][page][Hkv][row][dim], in order
    ramp = 0.05 + 6.0 * (torch.arange(69 * 16) / 1100.0) ** 2
    x["v_cache"] = (v * ramp.view(1, 69, 1, 16, 1)).view(-1, 2, 16, 128).to(torch.bfloat16)
    codes, scales = fp8_cache(x)
    got, err = run_fp8(x, codes, scales, num_splits=splits)
    assert err == 0
    assert_parity(got.cpu().numpy(), _want(x, codes, scales), f"G {G} S {splits}")
