"""The wide decode CTAs where the other tests do not reach: several runs of splits per unit in the layout of
two CTAs per SM, references that move late in each layout, error flags, and appended rows outside the
attended tokens. Everything against the fp64 oracle at the decode's tolerance."""
from __future__ import annotations

import math

import numpy as np
import pytest
import torch

import oracle
import paper_2606_21848_gb300 as kl
from paper_2606_21848_gb300.workloads import bf16_bits
from tests import _gpu
from tests._gpu import assert_parity, decode, oracle_decode, shape_of, to_dev
from tests._inputs import tiny

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    kl.build()
    kl.load()


# 320 units of 16 heads, more than two per SM: each split is a CTA. 3 and 8 states are merged by direct
# loads, 9 and 21 through the ring of three tiles.
@pytest.mark.parametrize("splits", [3, 8, 9, 21])
@pytest.mark.parametrize("G", [16, 11])
def test_runs_of_two_ctas_per_sm(splits, G):
    B, L = 320, splits * (384 if splits < 10 else 128)
    lens = tuple((L, L // 2 + 5, 129, 1, L - 128, 128, 0, 700)[i // 4 % 8] if i % 4 == 0 else 60 + i % 90
                 for i in range(B))
    x = tiny(B=B, Hq=G, Hkv=1, D=128, P=16, lens=lens, seed=230 + splits)
    assert kl.kl_decode_num_splits(shape_of(x), splits) == splits
    out, err = decode(to_dev(x), shape_of(x), num_splits=splits)
    assert err == 0
    assert_parity(out.cpu().numpy(), oracle_decode(x, _gpu.default_scale(x)), f"S {splits} G {G}")


# CTAs of 32 heads, of 16 with two softmax groups, and of 16 two to an SM
@pytest.mark.parametrize("B, G", [(80, 32), (2, 16), (160, 16)])
def test_reference_moves_late(B, G):
    """Rows that grow along 3000 tokens: a group's reference moves again after its sixth tile, with the
    sum of its earlier tiles and its last tile's output both in place."""
    L, pages = 3000, 188
    x = tiny(B=B, Hq=G, Hkv=1, D=128, P=16, lens=(L, L) + (1,) * (B - 2), seed=240 + G, table="identity")
    ramp = 0.05 + 6.0 * (torch.arange(pages * 16) / L) ** 2
    v = x["v_cache"].float()
    v[:2 * pages] *= ramp.view(pages, 1, 16, 1).repeat(2, 1, 1, 1)
    x["v_cache"] = v.to(torch.bfloat16)
    # largest score (base 2) of each head before token 12 * 128 and in the end: past the slack of 2^10
    q = torch.einsum("hk,kj->hj", x["q"][0].double(), x["w_r"][0].double())
    s = q @ x["v_cache"][:pages].double().reshape(-1, 128)[:L].T / math.sqrt(128) / math.log(2)
    assert float(((s.amax(-1) - s[:, :1536].amax(-1)) > 10).double().mean()) > 0.5
    out, err = decode(to_dev(x), shape_of(x), num_splits=1)
    assert err == 0
    assert_parity(out.cpu().numpy(), oracle_decode(x, _gpu.default_scale(x)), f"B {B} G {G}")


def _step(x, g, splits):
    B, Hq, D = x["q"].shape
    sh = shape_of(x)
    out = torch.full((B, Hq, D), float("nan"), dtype=torch.float32, device=_gpu.dev())
    err = torch.zeros(1, dtype=torch.int32, device=_gpu.dev())
    ws = torch.zeros(max(256, kl.kl_decode_workspace_size(sh, splits)), dtype=torch.uint8, device=_gpu.dev())
    kl.kl_decode_step(sh, g["q"], g["w_r"], g["v_new"], g["positions"], g["v_cache"], g["block_table"],
                      g["seq_lens"], kl.decode_options(splits), out, kl.KL_FP32, ws, err)
    torch.cuda.synchronize()
    return out, int(err.item())


@pytest.mark.parametrize("G", [16, 32])
@pytest.mark.parametrize("splits", [1, 3])
def test_append_outside_the_attended_tokens(G, splits):
    """The new row past the end of the sequence: in a tile that is read, in an empty run, and of a
    sequence without tokens."""
    B, held = 5, (800, 800, 800, 800, 800)
    x = tiny(B=B, Hq=2 * G, Hkv=2, D=128, P=16, lens=held, seed=250 + G)
    x["seq_lens"] = torch.tensor([130, 100, 0, 0, 500], dtype=torch.int32)
    x["positions"] = torch.tensor([200, 790, 0, 799, 500], dtype=torch.int32)
    g = to_dev(x)
    out, err = _step(x, g, splits)
    assert err == 0
    cache = oracle.append(bf16_bits(x["v_cache"]), bf16_bits(x["v_new"]), x["block_table"].numpy(),
                          x["positions"].numpy())
    np.testing.assert_array_equal(bf16_bits(g["v_cache"].cpu()), cache)
    x["v_cache"] = torch.from_numpy(cache.view(np.int16)).view(torch.bfloat16)
    assert_parity(out.cpu().numpy(), oracle_decode(x, _gpu.default_scale(x)), f"G {G} S {splits}")


@pytest.mark.parametrize("G", [16, 32])
@pytest.mark.parametrize("splits", [1, 3])
@pytest.mark.parametrize("fault, flag", [("page", kl.KL_FLAG_BAD_PAGE), ("no page", kl.KL_FLAG_BAD_PAGE),
                                         ("append page", kl.KL_FLAG_BAD_PAGE), ("length", kl.KL_FLAG_BAD_LENGTH),
                                         ("negative length", kl.KL_FLAG_BAD_LENGTH),
                                         ("position", kl.KL_FLAG_BAD_POSITION)])
def test_flags(G, splits, fault, flag):
    """A bad page, length or position of one sequence raises its flag, writes no other row and leaves
    the other sequences' outputs alone (all of them bounds-checked by the kernel)."""
    x = tiny(B=3, Hq=2 * G, Hkv=2, D=128, P=16, lens=(700, 800, 300), seed=260 + G)
    table = x["block_table"].clone()
    if fault == "page":
        table[1, 3] = x["num_pages"]
    elif fault == "no page":
        table[1, 3] = -1
    elif fault == "append page":
        x["seq_lens"][1], table[1, 49] = 700, x["num_pages"] + 5       # only the new row's page is bad
    elif fault == "length":
        x["seq_lens"][1] = table.shape[1] * 16 + 1
    elif fault == "negative length":
        x["seq_lens"][1] = -5
    else:
        x["positions"][1] = table.shape[1] * 16
    good = x["block_table"]
    x["block_table"] = table
    g = to_dev(x)
    out, err = _step(x, g, splits)
    assert err == flag
    x["block_table"] = good
    keep = [0, 2] if fault in ("page", "no page") else range(3)
    pos = x["positions"].clone()
    if fault in ("append page", "position"):           # no row of sequence 1: its own old row again
        pos[1] = 0
        page = int(good[1, 0])
        x["v_new"][1] = x["v_cache"][page, :, 0]
    cache = oracle.append(bf16_bits(x["v_cache"]), bf16_bits(x["v_new"]), good.numpy(), pos.numpy())
    np.testing.assert_array_equal(bf16_bits(g["v_cache"].cpu()), cache)
    x["v_cache"] = torch.from_numpy(cache.view(np.int16)).view(torch.bfloat16)
    if flag == kl.KL_FLAG_BAD_LENGTH:
        x["seq_lens"][1] = 0                            # taken as empty
    want = oracle_decode(x, _gpu.default_scale(x))
    got = out.cpu().numpy()
    for b in keep:
        assert_parity(got[b], want[b], f"{fault} G {G} S {splits} sequence {b}")
