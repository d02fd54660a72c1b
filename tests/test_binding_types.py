"""The binding takes and refuses what ctypes does for the same arguments (CPU only: every call is refused
by the host-side validation, or by the marshalling itself, before anything is launched)."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import paper_2606_21848_gb300 as kl


@pytest.fixture(scope="module", autouse=True)
def built():
    kl.build()


def _shape(cls=kl.kl_shape, num_seqs=2):
    return cls(num_seqs, 8, 2, 128, 16, 64, 32, 0, 0.0)


def _append(shape, v_new=16):
    kl.kl_append_v(shape, v_new, 16, 16, 16, None, 0)


def test_buffers_of_a_shapes_size_are_refused():
    n = ctypes.sizeof(kl.kl_shape)
    same = np.frombuffer(bytes(_shape(num_seqs=0)), np.int32)
    for bad in (bytes(n), bytearray(bytes(_shape(num_seqs=0))), memoryview(bytes(n)), same, None, 7):
        with pytest.raises(TypeError):
            _append(bad)

    class Alike(ctypes.Structure):
        _fields_ = kl.kl_shape._fields_

    for bad in (Alike(), (ctypes.c_int32 * 9)(), ctypes.pointer(_shape()), kl.decode_options()):
        with pytest.raises(ctypes.ArgumentError):
            _append(bad)
    for bad, error in ((bytes(ctypes.sizeof(kl.kl_decode_options)), TypeError), (_shape(), ctypes.ArgumentError)):
        with pytest.raises(error):
            kl.kl_decode_attention_ex(_shape(), 16, 16, 16, 16, 16, bad, 16, kl.KL_FP32, None, stream=0)
    with pytest.raises(ctypes.ArgumentError):
        kl.kl_latent_decode(_shape(), 16, 16, 16, 16, 16, 16, 0, 16, kl.KL_FP32, None, stream=0)


def test_a_shapes_subclass_is_a_shape():
    class More(kl.kl_shape):
        _fields_ = [("mine", ctypes.c_int64)]

    assert _append(More(0, 8, 2, 128, 16, 64, 32)) is None             # no sequences: nothing to do
    with pytest.raises(kl.KLError):
        _append(_shape(), 8)


class AsParameter:
    _as_parameter_ = ctypes.c_int32(-1)


@pytest.mark.parametrize("num", [-1, ctypes.c_int32(-1), ctypes.c_int(-1), AsParameter(), np.int32(-1),
                                 (1 << 32) - 1])
def test_integers(num):
    with pytest.raises(kl.KLError) as e:                   # a negative split count
        kl.kl_combine(_shape(), 16, 16, num, 16, kl.KL_FP32, stream=0)
    assert e.value.status == kl.KL_ERR_INVALID_ARG


@pytest.mark.parametrize("num", [None, 1.0, "1", ctypes.c_int64(1), ctypes.c_float(1), object()])
def test_other_numbers_are_refused(num):
    with pytest.raises(ctypes.ArgumentError):
        kl.kl_combine(_shape(num_seqs=0), 16, 16, num, 16, kl.KL_FP32, stream=0)


class Tensor:
    def __init__(self, addr):
        self.addr = addr

    def data_ptr(self):
        return self.addr


def test_addresses():
    with pytest.raises(kl.KLError):
        _append(_shape(), Tensor(None))                    # a null pointer
    for bad in (np.int64(16), 16.0, "16"):
        with pytest.raises(TypeError):
            _append(_shape(num_seqs=0), Tensor(bad))
