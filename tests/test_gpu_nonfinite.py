"""Infinities and NaN in cached rows, in the decodes whose softmax groups take alternate tiles. The wide
CTAs are compared with the sibling CTAs of 8 heads (one softmax state over all tiles; they serve the
same groups where the caller takes the split states): finite where those are finite, and equal
within the decode's tolerance, and not finite where those are not. A row whose score is -inf has
weight 0, also where it is all that a group's first tile holds."""
from __future__ import annotations

import math

import numpy as np
import pytest
import torch

import oracle
import paper_2606_21848_gb300 as kl
from paper_2606_21848_gb300.workloads import bf16_bits
from tests import _gpu
from tests._gpu import ATOL, RTOL, decode, shape_of, to_dev
from tests._inputs import tiny
from tests.test_gpu_fp8 import fp8_cache, run_fp8

pytestmark = pytest.mark.gpu

LENS = (129, 257, 130, 128, 300, 1, 385, 640)


@pytest.fixture(scope="module", autouse=True)
def lib():
    kl.build()
    kl.load()


def _put(x, b, t, dim, value):
    """value into dim `dim` of the row of token t of sequence b, every value head."""
    x["v_cache"][int(x["block_table"][b, t // 16]), :, t % 16, dim] = value


# CTAs of 16 heads two to an SM, of 32 heads, and of 16 heads with two softmax groups
@pytest.mark.parametrize("B, Hkv, G", [(24, 8, 16), (40, 4, 32), (8, 2, 16)])
@pytest.mark.parametrize("value", [math.inf, -math.inf, math.nan])
@pytest.mark.parametrize("last", [True, False])
def test_wide_like_siblings(B, Hkv, G, value, last):
    lens = (LENS * 5)[:B]
    x = tiny(B=B, Hq=Hkv * G, Hkv=Hkv, D=128, P=16, lens=lens, seed=210 + G)
    for b, L in enumerate(lens):
        if b % 3:                                    # every third sequence stays finite
            _put(x, b, L - 1 if last else L // 3, 7, value)
    for b, L in enumerate(lens):                     # a page's rows past the end may hold anything
        if L % 16:
            x["v_cache"][int(x["block_table"][b, L // 16]), :, L % 16:] = math.nan
    g, sh = to_dev(x), shape_of(x)
    wide, err = decode(g, sh, num_splits=1)
    assert err == 0
    part_o = torch.empty(B, Hkv * G, 1, 128, dtype=torch.float32, device=_gpu.dev())
    part_ml = torch.empty(B, Hkv * G, 1, 2, dtype=torch.float32, device=_gpu.dev())
    kl.kl_decode_attention_ex(sh, g["q"], g["w_r"], g["v_cache"], g["block_table"], g["seq_lens"],
                              kl.decode_options(1, partial_o=part_o, partial_ml=part_ml), None,
                              kl.KL_FP32, None)
    torch.cuda.synchronize()
    got, want = wide.cpu(), part_o[:, :, 0].cpu()
    fin = torch.isfinite(want)
    assert bool(fin.any()) and not bool(fin.all())
    assert torch.equal(torch.isfinite(got), fin), int((torch.isfinite(got) != fin).sum())
    assert bool(((got - want).abs() <= ATOL + RTOL * want.abs())[fin].all())


@pytest.mark.parametrize("G", [4, 8])
def test_fp8_overflowing_score(G):
    """The last token, alone in its tile, has a scale so large that its scores overflow: to -inf in
    about half of the heads, whose outputs are those of the other tokens."""
    x = tiny(B=3, Hq=2 * G, Hkv=2, D=128, P=16, lens=(129, 257, 385), seed=220)
    codes, scales = fp8_cache(x)
    for b, L in enumerate((129, 257, 385)):
        page = int(x["block_table"][b, (L - 1) // 16])
        codes[page, :, (L - 1) % 16] = 0x7E                    # 448 in every dim
        scales[page, :, (L - 1) % 16] = 3e38
    got, _ = run_fp8(x, codes, scales, num_splits=1)
    want = oracle.decode_fp8(bf16_bits(x["q"]), bf16_bits(x["w_r"]), codes, scales,
                             x["block_table"].numpy(), x["seq_lens"].numpy(), scale=1.0 / math.sqrt(128))
    low = np.abs(want).max(-1) < 1e30                          # heads whose score is -inf
    assert 0.2 < low.mean() < 0.8
    got = got.cpu().double().numpy()
    assert np.isfinite(got[low]).all()
    # (only there the group with the large scale has no other tile, whose output would be taken with that
    # scale's power of two)
    one = low.copy()
    one[1:] = False
    assert (np.abs(got - want)[one] <= ATOL + RTOL * np.abs(want[one])).all()
