"""Without Python's C headers the C module cannot be built: the library is, and the binding's functions go
through ctypes, with the same answers (CPU only)."""
from __future__ import annotations

import pytest

import paper_2606_21848_gb300 as kl
from paper_2606_21848_gb300 import _lib, builder
from tests import test_binding as same
from tests import test_binding_types as types


@pytest.fixture(autouse=True)
def no_headers(tmp_path, monkeypatch):
    kl.build()
    monkeypatch.setattr(builder, "PYMOD", str(tmp_path / "_keyless.so"))
    monkeypatch.setattr(builder, "python_headers", lambda: None)
    monkeypatch.setattr(_lib, "_native", None)


def test_build_needs_no_headers():
    assert builder.build() == builder.LIB
    assert isinstance(_lib._call(), _lib._Ctypes)


def test_a_module_left_out_by_mistake_is_reported(monkeypatch):
    monkeypatch.setattr(builder, "python_headers", lambda: "/usr/include")
    with pytest.raises(RuntimeError, match="not built"):
        _lib._call()


def test_same_answers():
    for stream in (0, same.Stream()):
        same.test_addresses_reach_the_library(stream)
    same.test_other_types_are_refused()
    same.test_options_and_keywords()
    types.test_buffers_of_a_shapes_size_are_refused()
    types.test_a_shapes_subclass_is_a_shape()
    types.test_addresses()
    for num in (-1, types.AsParameter()):
        types.test_integers(num)
    types.test_other_numbers_are_refused(1.0)


# one launching function of each argument pattern, refused by the library before any launch
def test_every_entry_point():
    s, z = kl.make_shape(2, 8, 2, 128, 16, 64, 32), kl.make_latent_shape(2, 8, 2, 128, 128, 16, 64, 32)
    calls = [(kl.kl_route_query, (s, None, 16, 16)), (kl.kl_append_v, (s, None, 16, 16, 16)),
             (kl.kl_decode_attention, (s, None, 16, 16, 16, 16, 0, 16, 0, None)),
             (kl.kl_decode_step, (s, 16, 16, None, 16, 16, 16, 16, None, 16, 0, None)),
             (kl.kl_combine, (s, None, 16, 1, 16, 0)),
             (kl.kl_standard_decode, (s, None, 16, 16, 16, 16, None, 16, 0, None)),
             (kl.kl_decode_attention_noalloc, (s, 16, 16, 16, 16, 16, -1, 16, 0)),
             (kl.kl_append_v_chunk, (s, None, 16, 16, 16, 4, 4, 16)),
             (kl.kl_append_v_fp8, (s, None, 16, 16, 16, 16)), (kl.kl_quantize_cache_fp8, (s, None, 16, 16)),
             (kl.kl_decode_step_fp8, (s, 16, 16, None, 16, 16, 16, 16, 16, 0, 16, 0, None)),
             (kl.kl_latent_decode_step, (z, 16, 16, 16, None, 16, 16, 16, 16, 0, 16, 0, None))]
    for f, args in calls:
        with pytest.raises(kl.KLError) as e:
            f(*args, stream=0)
        assert e.value.status == kl.KL_ERR_INVALID_ARG, f.__name__
