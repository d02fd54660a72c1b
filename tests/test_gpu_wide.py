"""GPU parity of the wide decode CTAs (16 or 32 query heads of a group per CTA, two softmax
groups taking alternate tiles) at the sizes where they can go wrong: 0, 1, 2 and 3 tiles with
every kind of remainder, groups that do not fill their heads, references that move, and runs of
splits merged inside the kernel. Everything against the fp64 oracle at the decode's tolerance.
"""
from __future__ import annotations

import pytest
import torch

import paper_2606_21848_gb300 as kl
from tests import _gpu
from tests._gpu import assert_parity, decode, oracle_decode, shape_of, to_dev
from tests._inputs import tiny

pytestmark = pytest.mark.gpu

EDGES = (0, 1, 15, 16, 17, 112, 127, 128, 129, 144, 255, 256, 257, 383, 384, 385, 500, 640, 641, 900)


@pytest.fixture(scope="module", autouse=True)
def lib():
    kl.build()
    kl.load()


# enough CTAs that groups of 17 and more take 32 heads per CTA (a wave of them), and few enough
# that they take 16
@pytest.mark.parametrize("B, Hkv, G, P", [(40, 4, 32, 16), (40, 4, 17, 32), (40, 4, 40, 128),
                                          (20, 1, 32, 16), (20, 2, 9, 64), (40, 8, 16, 16)])
@pytest.mark.parametrize("route", ["kv", "q", "none"])
def test_edges(B, Hkv, G, P, route):
    lens = (EDGES * 2)[:B]
    x = tiny(B=B, Hq=Hkv * G, Hkv=Hkv, D=128, P=P, lens=lens, seed=60 + G,
             wr_per_query_head=route == "q")
    g = to_dev(x)
    if route == "none":
        g["w_r"] = None
        x["w_r"] = torch.eye(128).expand(Hkv, 128, 128).contiguous().to(torch.bfloat16)
    out, err = decode(g, shape_of(x), num_splits=1)
    assert err == 0
    assert_parity(out.cpu().numpy(), oracle_decode(x, _gpu.default_scale(x)), f"{B} {Hkv} {G} {route}")


@pytest.mark.parametrize("Hkv, G", [(8, 16), (8, 32)])
def test_moving_reference(Hkv, G):
    """Rows that grow along the sequence: scores pass the running reference by more than the slack
    several times, so O and the sums are rescaled with tiles already accumulated."""
    x = tiny(B=20, Hq=Hkv * G, Hkv=Hkv, D=128, P=16, lens=(1100,) * 20, seed=70, table="identity")
    v = x["v_cache"].float()                       # [20 * 69 pages][Hkv][16][128], in token order
    ramp = 0.05 + 6.0 * (torch.arange(69 * 16) / 1100.0) ** 2
    v = v.view(20, 69, Hkv, 16, 128) * ramp.view(1, 69, 1, 16, 1)
    x["v_cache"] = v.view(-1, Hkv, 16, 128).to(torch.bfloat16)
    out, err = decode(to_dev(x), shape_of(x), num_splits=1)
    assert err == 0
    assert_parity(out.cpu().numpy(), oracle_decode(x, _gpu.default_scale(x)), f"G {G}")


@pytest.mark.parametrize("G, splits", [(32, 300), (32, 3), (12, 70)])
def test_runs_merged(G, splits):
    x = tiny(B=1, Hq=G, Hkv=1, D=128, P=16, lens=(40000,), seed=80 + G)
    out, err = decode(to_dev(x), shape_of(x), num_splits=splits, out_dtype=kl.KL_BF16)
    assert err == 0
    assert_parity(out.float().cpu().numpy(), oracle_decode(x, _gpu.default_scale(x)), f"S {splits}")


# CTAs of 32 heads that leave SMs idle: CTAs of 16 would share SMs (the first three) or run more
# splits each (the last two)
@pytest.mark.parametrize("B, Hkv, G, P, splits", [(77, 1, 32, 16, 1), (60, 1, 40, 16, 1),
                                                  (151, 1, 17, 64, 1), (30, 1, 32, 16, 4),
                                                  (19, 2, 24, 32, 3)])
def test_partly_filled_wave(B, Hkv, G, P, splits):
    lens = (EDGES * 8)[:B]
    x = tiny(B=B, Hq=Hkv * G, Hkv=Hkv, D=128, P=P, lens=lens, seed=90 + G)
    out, err = decode(to_dev(x), shape_of(x), num_splits=splits)
    assert err == 0
    assert_parity(out.cpu().numpy(), oracle_decode(x, _gpu.default_scale(x)), f"{B} {G} S {splits}")
