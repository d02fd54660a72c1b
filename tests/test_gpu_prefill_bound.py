"""Prefills whose host bound on the chunk length is large (it sizes the grid; short chunks may come with
a loose one): the layout chosen for the bound must be one that can be launched."""
from __future__ import annotations

import math

import pytest

from tests._gpu import assert_parity
from tests._inputs import tiny_prefill
from tests.test_gpu_prefill import lib, oracle_prefill, run_prefill  # noqa: F401 (lib: fixture)

pytestmark = pytest.mark.gpu


# bounds around those where 64, 32 and 16 heads per block would pass the grid's z extent
@pytest.mark.parametrize("G, bound", [(64, 131070), (64, 131073), (32, 262145), (16, 524290), (1, 65535 * 128)])
def test_loose_bound(G, bound):
    x = tiny_prefill(B=2, Hq=G, Hkv=1, D=128, P=16, lens=(300, 40), q_lens=(5, 40), seed=160)
    got, err = run_prefill(x, max_q=bound)
    assert err == 0
    assert_parity(got.float().cpu().numpy(), oracle_prefill(x, 1.0 / math.sqrt(128)), f"G {G} bound {bound}")
