"""GPU parity of the chunked prefill at the edges of its 64-token half tiles: every remainder
around one to five half tiles, odd and even counts, chunks that end mid-block, and references
that move while half tiles of both softmax groups are in flight."""
from __future__ import annotations

import math

import pytest
import torch

from tests._gpu import assert_parity
from tests._inputs import tiny_prefill
from tests.test_gpu_prefill import lib, oracle_prefill, run_prefill  # noqa: F401 (lib: fixture)

pytestmark = pytest.mark.gpu

EDGES = (1, 63, 64, 65, 127, 128, 129, 191, 192, 193, 255, 256, 257, 320, 321)


@pytest.mark.parametrize("chunk", [1, 2, 64, 129, 400])
def test_half_tile_edges(chunk):
    x = tiny_prefill(B=len(EDGES), Hq=4, Hkv=2, D=128, P=16, lens=EDGES,
                     q_lens=tuple(min(chunk, n) for n in EDGES), seed=90 + chunk)
    got, err = run_prefill(x)
    assert err == 0
    assert_parity(got.cpu().numpy(), oracle_prefill(x, 1.0 / math.sqrt(128)), f"chunk {chunk}")


@pytest.mark.parametrize("chunk", [130, 900])
def test_moving_reference(chunk):
    """Rows that grow along the sequence: the reference moves by more than 2^8 several times."""
    x = tiny_prefill(B=2, Hq=4, Hkv=2, D=128, P=16, lens=(900, 900), q_lens=(chunk, chunk), seed=95,
                     table="identity")
    v = x["v_cache"].float().view(2, 57, 2, 16, 128)      # [b][page][Hkv][row][dim], in order
    ramp = 0.05 + 6.0 * (torch.arange(57 * 16) / 900.0) ** 2
    x["v_cache"] = (v * ramp.view(1, 57, 1, 16, 1)).view(-1, 2, 16, 128).to(torch.bfloat16)
    got, err = run_prefill(x)
    assert err == 0
    assert_parity(got.cpu().numpy(), oracle_prefill(x, 1.0 / math.sqrt(128)), f"chunk {chunk}")
