"""Arguments of the binding's calls: what ctypes refuses is refused, what it converts is converted the same way, and nothing
reaches the library in another argument's place (no GPU needed: the called library is a stub that records its arguments)."""
import ctypes
import platform
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2110_15362_b200 import binding as B
from paper_2110_15362_b200 import build

WORDS = 18
N = 5000


@pytest.fixture(scope="module", params=["x86_64", "aarch64"])
def stub(tmp_path_factory, request):
    """A library with the exported names, opened as a build of the product library; every function records what it gets.
    On a host that the native call path is not for, the binding calls through ctypes alone."""
    d = tmp_path_factory.mktemp("stub")
    args = ", ".join("W a%d" % k for k in range(WORDS))
    lines = ["typedef unsigned long long W;", "W seen[%d], called; float f_seen;" % WORDS]
    for name in B.EXPORTS:
        if name in B.CALLS:
            lines.append("int %s(%s, float f) { W v[] = {%s}; for (int k = 0; k < %d; ++k) seen[k] = v[k]; f_seen = f; ++called; return 0; }"
                         % (name, args, ", ".join("a%d" % k for k in range(WORDS)), WORDS))
        else:
            lines.append("int %s(void) { return 0; }" % name)
    (d / "s.c").write_text("\n".join(lines))
    subprocess.check_call(["gcc", "-O1", "-shared", "-fPIC", "-o", str(d / "s.so"), str(d / "s.c")])
    with pytest.MonkeyPatch.context() as m:
        m.setattr(platform, "machine", lambda: request.param)
        if request.param != "x86_64":                # nothing is compiled or loaded there
            m.setattr(subprocess, "check_call", None)
            m.setitem(sys.modules, "paper_2110_15362_b200._pycall", None)
        build.build_caller(force=request.param != "x86_64")
        return B.load_library(str(d / "s.so"))


@pytest.fixture
def S(stub, monkeypatch):
    monkeypatch.setattr(B, "_lib", stub)
    monkeypatch.setattr(B, "_stream", lambda stream: 0x77)
    stub.words = (ctypes.c_uint64 * WORDS).in_dll(stub, "seen")
    stub.float = ctypes.c_float.in_dll(stub, "f_seen")
    stub.count = ctypes.c_uint64.in_dll(stub, "called")
    stub.count.value = 0
    return stub


def _buffers():
    return [torch.zeros(64) for _ in range(6)]


def _compress(n=None, capacity=None, dense=None, bitmap=None):
    x, bm, values, prefix, nnz, ws = _buffers()
    dense, bitmap = x if dense is None else dense, bm if bitmap is None else bitmap
    B.bt_compress(dense, bitmap, values, prefix, nnz, ws, None, n=n, values_capacity=capacity)
    return [dense.data_ptr(), n, B.BT_F32, bitmap.data_ptr(), values.data_ptr(), capacity, prefix.data_ptr(), nnz.data_ptr(), ws.data_ptr(),
            256, 0, 0x77]


class _Index:
    def __index__(self):
        return 41


COUNTS = [(0, 0), (N, N), (1 << 63, 1 << 63), (-2, (1 << 64) - 2), (True, 1), (np.int64(77), 77), (np.uint32(9), 9), (torch.tensor([33]), 33),
          (torch.tensor(34), 34), (ctypes.c_uint64(35), 35), (_Index(), 41)]


@pytest.mark.parametrize("given,taken", COUNTS)
def test_counts_are_taken_by_value(S, given, taken):
    want = _compress(given, given)
    want[1] = want[5] = taken
    assert list(S.words)[:12] == want and S.count.value == 1


@pytest.mark.parametrize("given", [0.5, float(N), np.float64(3.0), np.float32(3.0), torch.tensor([1, 2]), torch.tensor(1.5), "12", b"12", np.zeros(3),
                                   (ctypes.c_uint64 * 2)(), ctypes.c_int(3)])
@pytest.mark.parametrize("where", ["n", "capacity"])
def test_what_is_no_count_is_refused(S, given, where):
    with pytest.raises((TypeError, ctypes.ArgumentError)):
        _compress(**{"n": 64, "capacity": 64, where: given})
    assert S.count.value == 0


@pytest.mark.parametrize("given", [0x10000, 1.5, np.zeros(64), (ctypes.c_uint64 * 2)(), "x", b"xxxxxxxx"])
@pytest.mark.parametrize("call", ["compress", "mask", "pool", "arena_batch"])
def test_what_is_no_tensor_is_refused(S, given, call):
    x, bm, values, prefix, nnz, ws = _buffers()
    with pytest.raises(AttributeError):
        if call == "compress":
            B.bt_compress(x, given, values, prefix, nnz, ws, n=64)
        elif call == "mask":
            B.bt_mask_compress(x, bm, given, None, values)
        elif call == "pool":
            B.bt_maxpool2x2_fwd(x, given, None, planes=1, height=8, width=8)
        else:
            B.bt_compress_arena_batch((B.BatchItem * 1)(), torch.float32, x, given, prefix, ws)
    assert S.count.value == 0


@pytest.mark.parametrize("tau,taken", [(0.5, 0.5), (3, 3.0), (True, 1.0), (np.float32(0.25), 0.25), (np.float64(0.25), 0.25), (torch.tensor(0.75), 0.75)])
def test_thresholds_are_taken_as_floats(S, tau, taken):
    x, bm, values, prefix, nnz, ws = _buffers()
    B.bt_prune_fwd_compress(x, tau, None, bm, values, prefix, nnz, ws)
    assert S.float.value == taken and S.count.value == 1
    assert list(S.words)[:4] == [x.data_ptr(), 64, B.BT_F32, 0]                   # nothing moved up or down a place
    assert S.words[5] == values.data_ptr() and S.words[6] == 64 and S.words[11] == 0 and S.words[12] == 0x77


@pytest.mark.parametrize("tau", ["0.5", None, b"1", [0.5]])
def test_what_is_no_threshold_is_refused(S, tau):
    x, bm, values, prefix, nnz, ws = _buffers()
    for call in (lambda: B.bt_prune_fwd_compress(x, tau, None, bm, values, prefix, nnz, ws),
                 lambda: B.bt_prune_fwd_compress_arena(x, tau, None, bm, ws, nnz, nnz, prefix, nnz, ws)):
        with pytest.raises((TypeError, ctypes.ArgumentError)):
            call()
    assert S.count.value == 0


class _OtherItem(ctypes.Structure):
    _fields_ = B.BatchItem._fields_


@pytest.mark.parametrize("items", [np.zeros(9, np.uint64), (ctypes.c_uint64 * 9)(), (_OtherItem * 1)(), torch.zeros(9), b"0" * 72, [B.BatchItem()]])
def test_what_is_no_batch_is_refused(S, items):
    with pytest.raises((TypeError, ctypes.ArgumentError)):
        B.bt_decompress_batch(items, torch.float32)
    assert S.count.value == 0


def test_batches_are_taken(S):
    items = (B.BatchItem * 3)()
    B.bt_decompress_batch(items, torch.float32)
    assert list(S.words)[:4] == [ctypes.addressof(items), 3, B.BT_F32, 0x77]


def test_the_number_of_arguments_is_checked(S):
    x = torch.zeros(64)
    for calls in (S.calls, S.tensor_calls):
        with pytest.raises((TypeError, ctypes.ArgumentError)):
            calls.bt_compress(x, 64, B.BT_F32)
        with pytest.raises((TypeError, ctypes.ArgumentError)):
            calls.bt_decompress(x, x, x, 64, B.BT_F32, x)
    assert S.count.value == 0


@pytest.mark.parametrize("name", B.CALLS)
def test_every_call_passes_what_ctypes_passes(S, name):
    """Distinct ordinary values for every parameter, through each wrapped form and through ctypes."""
    u64, i32, u32 = ctypes.c_uint64, ctypes.c_int, ctypes.c_uint32
    fn = getattr(S, name)
    plain, wrapped, with_addresses = [], [], []
    for k, t in enumerate(fn.argtypes):
        last = k + 1 == len(fn.argtypes)
        if t is ctypes.c_void_p and not last:
            v = torch.zeros(16) if k % 3 else None
            at = None if v is None else v.data_ptr()
            plain.append(at), wrapped.append(v), with_addresses.append(at)
            continue
        v = (B.BatchItem * 2)() if t is ctypes.POINTER(B.BatchItem) else 0.375 if t is ctypes.c_float else {u64: (1 << 63) + 3 * k, i32: 5 + k, u32: 9 + k}.get(t, 0x1000 + k)
        plain.append(v), wrapped.append(v), with_addresses.append(v)
    seen = []
    for call, args in ((fn, plain), (getattr(S.tensor_calls, name), wrapped), (getattr(S.calls, name), wrapped), (getattr(S.calls, name), with_addresses)):
        assert call(*args) == 0
        words = sum(t is not ctypes.c_float for t in fn.argtypes)
        seen.append((list(S.words)[:words], S.float.value if ctypes.c_float in fn.argtypes else None))
        assert len(seen[0][0]) + (seen[0][1] is not None) == len(fn.argtypes)
    assert seen.count(seen[0]) == 4
