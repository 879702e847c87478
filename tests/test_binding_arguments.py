"""What the Python entry points take for an argument, as far as it shows without a GPU: every call here is refused
before the library is entered (the parameters are CPU tensors)."""
import ctypes
import types

import pytest
import torch

import paper_1610_02132_b200 as Q

X = torch.zeros(64)
BYTES = torch.zeros(256, dtype=torch.uint8)
STATUS = torch.zeros(1, dtype=torch.int32)
NOT_ON_GPU = "must be a contiguous CUDA tensor"


def decode(msgs=(BYTES,), tables=(BYTES,), status=STATUS, payload_bytes=None, packed=False, n=64):
    if packed:
        Q.qsgd_decode_accumulate_packed(msgs, tables, n, 32, 15, Q.CODE_ELIAS, X, status, msg_bytes=payload_bytes)
    else:
        Q.qsgd_decode_accumulate(msgs, tables, n, 32, 15, Q.CODE_ELIAS, X, status, payload_bytes=payload_bytes)


@pytest.mark.parametrize("bad", [4096, True, object()])
def test_status_and_workspace_are_tensors_not_addresses(bad):
    with pytest.raises(AttributeError, match="data_ptr"):
        decode(status=bad)
    with pytest.raises(AttributeError, match="data_ptr"):
        Q.qsgd_encode(X, 32, 15, Q.NORM_L2, Q.CODE_ELIAS, 7, 0, 0, BYTES, BYTES, bad, STATUS)
    with pytest.raises(AttributeError, match="data_ptr"):
        decode(status=None)


def test_storages_and_other_holders_of_a_data_ptr_are_taken():
    holder = types.SimpleNamespace(data_ptr=lambda: 4096)
    for msg in (BYTES, BYTES.untyped_storage(), holder, 4096):
        with pytest.raises(Q.QsgdError, match=NOT_ON_GPU):
            decode(msgs=[msg], tables=[msg], status=STATUS)
    with pytest.raises(Q.QsgdError, match=NOT_ON_GPU):
        decode(status=STATUS.untyped_storage())


def test_numbers_of_ctypes_are_taken():
    native = Q.binding._native
    native.encode                                          # loads the module
    native = Q.binding._native
    for n, eta in ((ctypes.c_uint64(64), ctypes.c_float(0.5)), (64, 1)):
        with pytest.raises(Q.QsgdError, match="x " + NOT_ON_GPU):
            native.decode(False, [4096], [4096], None, n, 32, 15, 1, X, eta, STATUS, None)
    for n in (1.5, "64", None):
        with pytest.raises(TypeError):
            native.decode(False, [4096], [4096], None, n, 32, 15, 1, X, 0.5, STATUS, None)


def test_lists_of_messages_have_a_length():
    """A generator would be used up by the first of its two readings: the packed form then took every message for
    empty."""
    for bad in ((m for m in [BYTES]), iter([BYTES]), 7):
        with pytest.raises(TypeError):
            decode(msgs=bad, packed=True)
    for good in ([BYTES], (BYTES,), {0: 4096}.values()):
        with pytest.raises(Q.QsgdError, match=NOT_ON_GPU):
            decode(msgs=good, payload_bytes=[256], packed=True)
