"""What the Python entry points take for an argument, as far as it shows without a GPU: every call here is refused
before the library is entered (the parameters are CPU tensors)."""
import ctypes
import os
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


@pytest.mark.parametrize("packed", [False, True])
def test_too_few_tables_or_byte_counts(packed):
    """What is missing read as a bound that was not given, and the payloads were then read without one."""
    two = [4096, 8192]
    for kw in (dict(tables=[4096], payload_bytes=[64, 64]), dict(tables=two, payload_bytes=[64]),
               dict(tables=two, payload_bytes=[])):
        with pytest.raises(Q.QsgdError, match="given for 2 messages"):
            decode(msgs=two, packed=packed, **kw)
    decoded = dict(msgs=two, tables=two + [16], payload_bytes=[64, 64, 64], packed=packed)      # more are no harm
    with pytest.raises(Q.QsgdError, match=NOT_ON_GPU):
        decode(**decoded)
    native = Q.binding._native
    for code in (Q.CODE_FIXED, 9):                         # no tables there (9: the library refuses it)
        with pytest.raises(Q.QsgdError, match=NOT_ON_GPU):
            native.decode(packed, two, [], [], 64, 32, 15, code, X, None, STATUS, None)


def test_too_few_tables_or_byte_counts_under_policy():
    native, two = Q.binding._native, [4096, 8192]
    for n_buckets, refused in ((2, True), (0, False)):     # raw tensors alone have no tables
        plan = Q.binding.PolicyStruct(16, 16, n_buckets, 16, 16, 1, 8, 72, 1)
        for tables, counts in (([4096], None), (two, [64])):
            with pytest.raises(Q.QsgdError, match="given for 2 messages" if refused else NOT_ON_GPU):
                native.policy_decode(two, tables, counts, ctypes.addressof(plan), 32, 15, Q.CODE_ELIAS, X, None, STATUS,
                                     None)


def test_policy_calls_hand_over_the_struct_that_the_plan_has_now(monkeypatch):
    seen = []
    native = types.SimpleNamespace(policy_decode=lambda *a: seen.append(a[3]) or 0)
    monkeypatch.setattr(Q.binding, "_native", native)
    monkeypatch.setattr(Q.binding, "_covered", lambda *a: None)
    plan = types.SimpleNamespace(bucket=32, n=64)
    structs = [Q.binding.PolicyStruct() for _ in range(2)]
    for plan.struct in structs:
        Q.qsgd_policy_decode_accumulate([4096], None, plan, 15, Q.CODE_FIXED, X, STATUS)
        Q.qsgd_policy_decode_sgd_step([4096], None, plan, 15, Q.CODE_FIXED, X, 0.5, STATUS)
    assert seen == [ctypes.addressof(s) for s in structs for _ in range(2)]


def test_native_module_belongs_to_the_torch_and_python_that_run(monkeypatch):
    """It reads torch's objects directly: one compiled against another torch or Python must not be loaded."""
    from paper_1610_02132_b200 import build
    build.build()
    mine = build.native_path()
    assert os.path.exists(mine)
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert build.native_path() != mine
    with pytest.raises(Q.QsgdError, match="not built"):
        Q.binding._Native().encode
    monkeypatch.undo()
    monkeypatch.setattr("sysconfig.get_config_var", lambda name: ".cpython-30.so")
    assert build.native_path() != mine
