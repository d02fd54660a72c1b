"""Argument marshalling of the binding's C module (CPU only: every call is refused by the host-side
validation, or by the marshalling itself, before anything is launched)."""
from __future__ import annotations

import ctypes

import pytest

import paper_2606_21848_gb300 as kl


@pytest.fixture(scope="module", autouse=True)
def built():
    kl.build()


def _shape(**kw):
    d = dict(num_seqs=2, num_q_heads=8, num_kv_heads=2, head_dim=128, page_size=16, num_pages=64,
             max_pages_per_seq=32)
    d.update(kw)
    return kl.make_shape(**d)


class Tensor:
    def __init__(self, addr):
        self.addr = addr

    def data_ptr(self):
        return self.addr


class Stream:
    cuda_stream = 0


def _append(shape, v_new, **kw):
    kl.kl_append_v(shape, v_new, 16, 16, kw.get("cache", 16), None, kw.get("stream", 0))


@pytest.mark.parametrize("stream", [0, Stream()])
def test_addresses_reach_the_library(stream):
    for bad in (None, 0, Tensor(0), 8, Tensor(8)):         # null, then misaligned
        with pytest.raises(kl.KLError) as e:
            _append(_shape(), bad, stream=stream)
        assert e.value.status == kl.KL_ERR_INVALID_ARG
    assert _append(_shape(num_seqs=0), Tensor(16), stream=stream) is None   # nothing to do


def test_other_types_are_refused():
    with pytest.raises(ctypes.ArgumentError):
        _append(kl.make_latent_shape(2, 8, 2, 128, 128, 16, 64, 32), 16)
    with pytest.raises(TypeError):
        _append("shape", 16)
    with pytest.raises(AttributeError):
        _append(_shape(), object())
    with pytest.raises(AttributeError):
        _append(_shape(), 16, stream=object())
    with pytest.raises(ctypes.ArgumentError):
        kl.kl_combine(_shape(), 16, 16, 2.0, 16, kl.KL_FP32, stream=0)


def test_options_and_keywords():
    with pytest.raises(kl.KLError) as e:                   # negative split count, from the structure
        kl.kl_decode_attention_ex(shape=_shape(), q=16, w_r=16, v_cache=16, block_table=16, seq_lens=16,
                                  opts=kl.decode_options(-1), out=16, out_dtype=kl.KL_FP32,
                                  workspace=None, err=None, stream=0)
    assert e.value.status == kl.KL_ERR_INVALID_ARG
    with pytest.raises(kl.KLError) as e:                   # None: the defaults, which need a workspace
        kl.kl_decode_attention_ex(_shape(max_pages_per_seq=2048), 16, 16, 16, 16, 16, None, 16,
                                  kl.KL_FP32, None, stream=0)
    assert e.value.status == kl.KL_ERR_WORKSPACE
