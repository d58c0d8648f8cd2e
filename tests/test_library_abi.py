"""Host-side checks of the CUDA library that need no GPU: it loads, exports every
symbol the public header declares, and its pure host entry points behave."""
import ctypes as C
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def qesgd():
    from paper_1901_03040_b200 import build
    build.build()
    from paper_1901_03040_b200 import qesgd as mod
    return mod


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "qesgd.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(qesgd_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported_and_bound(qesgd):
    names = _declared_symbols()
    assert len(names) >= 16
    for name in names:
        assert hasattr(qesgd.lib, name), f"{name} is declared in qesgd.h but not exported"
        assert name in qesgd.SIGNATURES, f"{name} has no ctypes signature"
    assert sorted(qesgd.SIGNATURES) == names


def test_size_helpers(qesgd):
    assert qesgd.num_buckets(0, 512) == 0
    assert qesgd.num_buckets(1, 512) == 1
    assert qesgd.num_buckets(11_689_512, 512) == 22_832
    assert qesgd.num_buckets(25_557_032, 256) == 99_833
    assert qesgd.num_buckets(1 << 30, 128) == 8_388_608
    assert qesgd.num_buckets(100, 100) == 0            # not a power of two
    assert qesgd.code_bytes(1 << 24, 512, 2) == 4 << 20
    assert qesgd.code_bytes(1 << 24, 512, 8) == 16 << 20
    assert qesgd.code_bytes(11_689_512, 512, 4) == 22_832 * 256
    assert qesgd.code_bytes(1000, 512, 3) == 0
    for bucket in (64, 128, 8192):
        for bits in (2, 4, 8):
            assert qesgd.code_bytes(12345, bucket, bits) % 16 == 0


def test_null_context_and_strerror(qesgd):
    lib = qesgd.lib
    assert lib.qesgd_destroy(None) == qesgd.EINVAL
    assert lib.qesgd_encode(None, None, None, 10, 512, 7, 4, 0, 0.0, 0, 0, 0, None, None) == qesgd.EINVAL
    assert lib.qesgd_decode(None, None, None, 10, 512, 7, 4, None) == qesgd.EINVAL
    assert lib.qesgd_status(None, None) == qesgd.EINVAL
    assert lib.qesgd_launch_count(None) == 0
    assert lib.qesgd_strerror(0) == b"ok"
    assert b"invalid" in lib.qesgd_strerror(qesgd.EINVAL)
    assert lib.qesgd_create(None, 0, None) == qesgd.EINVAL
    assert lib.qesgd_set_wait_limit(None, 1000) == qesgd.EINVAL
    assert lib.qesgd_debug_drop_signal(None, 0) == qesgd.EINVAL
    assert lib.qesgd_debug_lr_plan(None, None) == qesgd.EINVAL


def test_create_without_a_device_fails_cleanly(qesgd):
    import torch
    if torch.cuda.is_available():
        pytest.skip("a device is present")
    handle = C.c_void_p()
    rc = qesgd.lib.qesgd_create(C.byref(handle), 0, None)
    assert rc in (qesgd.ECUDA, qesgd.EINVAL) and not handle.value


class _WithIndex:
    def __index__(self):
        return 5


class _AsParameter:
    _as_parameter_ = 5


class _Tensor:
    def __init__(self, address):
        self.address = address

    def data_ptr(self):
        return self.address


# a size, a count, a float and a tensor in every form that ctypes converts or refuses
_FORMS = [("d", v) for v in (5, True, -1, 1 << 70, "numpy.int64", "numpy.uint32", "tensor", "array", _WithIndex(), C.c_uint64(5),
                             C.c_uint32(5), _AsParameter(), 5.0, "5", None)]
_FORMS += [("batch", v) for v in (5, (1 << 32) + 5, "numpy.int64", C.c_uint32(5), C.c_uint64(5), 5.0)]
_FORMS += [("lr", v) for v in (1, 0.5, 1e300, 10 ** 400, "numpy.float32", "ftensor", C.c_float(0.5), C.c_double(0.5), "1", None)]
_FORMS += [("u", v) for v in (None, _Tensor(4096), _Tensor(None), _Tensor(5.0), _Tensor(True), 4096)]


@pytest.mark.parametrize("slot,value", _FORMS, ids=[f"{s}-{v!r}"[:40] if isinstance(v, (int, float, str, type(None))) else
                                                    f"{s}-{type(v).__name__}" for s, v in _FORMS])
def test_the_binding_converts_arguments_as_ctypes_does(qesgd, slot, value):
    """qesgd_lr_local_epoch with one argument in some other form than int, float or tensor: the library
    receives what ctypes makes of it, and what ctypes refuses is refused with the same exception."""
    import numpy as np
    import torch
    made = {"numpy.int64": np.int64(5), "numpy.uint32": np.uint32(5), "tensor": torch.tensor(5), "array": np.array(5),
            "numpy.float32": np.float32(0.5), "ftensor": torch.tensor(0.5)}
    value = made.get(value, value) if isinstance(value, str) else value
    name = "qesgd_lr_local_epoch"
    res, kinds = qesgd.SIGNATURES[name]
    seen = []
    callback = C.CFUNCTYPE(res, *kinds)(lambda *a: seen.append(a) or qesgd.OK)
    call = dict(X=None, y=None, n_local=7, d=64, batch=3, lr=0.25, u=None)
    call[slot] = value

    def outcome(run):
        seen.clear()
        try:
            run()
        except Exception as e:                       # noqa: BLE001  (the kind of exception is what is compared)
            return type(e), None
        return None, list(seen)

    def through_ctypes():
        args = [call["X"], call["y"], call["n_local"], call["d"], call["batch"], call["lr"]]
        C.CFUNCTYPE(res, *kinds)(C.cast(callback, C.c_void_p).value)(
            None, *args, None if call["u"] is None else C.c_void_p(call["u"].data_ptr()))

    ctx = qesgd.Context.__new__(qesgd.Context)
    ctx._h, ctx._address = None, 0
    table = {n: C.cast(getattr(qesgd.lib, n), C.c_void_p).value for n in qesgd.SIGNATURES}

    def by_ctypes(n, args):
        return C.CFUNCTYPE(res, *kinds)(C.cast(callback, C.c_void_p).value)(C.c_void_p(args[0]), *[
            C.c_void_p(a.data_ptr()) if k is C.c_void_p and a is not None else a for k, a in zip(kinds[1:], args[1:])])
    qesgd._native.bind({**table, name: C.cast(callback, C.c_void_p).value}, by_ctypes)
    try:
        got = outcome(lambda: ctx.qesgd_lr_local_epoch(**call))
    finally:
        qesgd._native.bind(table, qesgd._by_ctypes)
    want = outcome(through_ctypes)
    assert got == want
    assert want[0] is not None or len(want[1]) == 1
    # the table as the module binds it: without a context every accepted form is an invalid argument
    if want[0] is None:
        with pytest.raises(qesgd.QesgdError):
            ctx.qesgd_lr_local_epoch(**call)
    else:
        with pytest.raises(want[0]):
            ctx.qesgd_lr_local_epoch(**call)
