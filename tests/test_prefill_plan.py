"""The chunked prefill's launch layout (csrc/kl_prefill_plan.cuh), compiled for the host: heads per
block, rows per block and CTAs per cluster around the sizes where the rules change, and a grid that
the hardware takes for every chunk that the entry point accepts."""
from __future__ import annotations

import ctypes
import os
import subprocess

import pytest

from paper_2606_21848_gb300 import builder

GRID_Z = 65535            # largest z extent of a grid
MAX_Q = GRID_Z * 128      # longest chunk that kl_prefill_attention accepts
SRC = """
#include "kl_prefill_plan.cuh"
extern "C" void plan(int B, int Hkv, int G, int max_q, long long max_tokens, int per_q, int sms, int *out) {
    const kl::PrefillPlan p = kl::plan_prefill(B, Hkv, G, max_q, max_tokens, per_q != 0, sms);
    out[0] = p.hp; out[1] = p.rpb; out[2] = p.cs;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SRC)
    lib = str(d / "plan.so")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-shared", "-fPIC", "-I", builder.CSRC,
                    str(d / "plan.cpp"), "-o", lib], check=True)
    f = ctypes.CDLL(lib).plan
    f.argtypes = [ctypes.c_int] * 4 + [ctypes.c_longlong, ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]

    def call(B, Hkv, G, max_q, max_tokens=None, per_q=False, sms=152):
        out = (ctypes.c_int * 3)()
        f(B, Hkv, G, max_q, max_tokens or max(max_q, 8192), int(per_q), sms, out)
        return tuple(out)
    return call


@pytest.mark.parametrize("G", [1, 2, 3, 7, 8, 12, 16, 32, 64, 71, 128])
def test_every_accepted_chunk_fits_the_grid(plan, G):
    sizes = {MAX_Q}
    for hp in (1, 2, 4, 8, 16, 32, 64):
        for blocks in (1, 2, 513, 1024, 1025, GRID_Z - 1, GRID_Z, GRID_Z + 1):
            sizes.update(blocks * (128 // hp) + k for k in (-1, 0, 1, 2))
    for max_q in sorted(n for n in sizes if 1 <= n <= MAX_Q):
        hp, rpb, cs = plan(1, 1, G, max_q)
        assert 1 <= hp <= min(G, 64) and rpb == 128 // hp and cs in (1, 2, 4, 8), (max_q, hp, rpb, cs)
        assert -(-max_q // rpb) <= GRID_Z, (max_q, hp)
        # never more blocks than with one head each
        assert -(-G // hp) * -(-max_q // rpb) <= G * -(-max_q // 128), (max_q, hp)
        assert plan(1, 1, G, max_q, per_q=True)[:2] == (1, 128)


@pytest.mark.parametrize("args, want", [
    ((1, 1, 64, 131072), (1, 128, 1)), ((1, 1, 64, 131070), (64, 2, 1)),   # 65535 blocks of 64 heads
    ((1, 8, 4, 512), (1, 128, 1)), ((16, 8, 4, 1, 512), (4, 32, 1)),
    ((4, 2, 6, 16, 4096), (6, 21, 8)), ((2, 8, 4, 100, 8192), (1, 128, 2)),
    ((1, 1, 2, 60, 2000), (2, 64, 8)), ((70, 1, 2, 60, 2048), (2, 64, 2)), ((100, 1, 2, 60, 2048), (2, 64, 1))])
def test_layouts(plan, args, want):
    assert plan(*args) == want
