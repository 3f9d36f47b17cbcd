"""The extension the binding calls the library through (csrc/bt_pycall.c), functions wrapped without their parameters'
kinds: every kind of argument, in registers and on the stack, arrives where the called function expects it (no GPU needed:
the called functions are compiled here).  What a wrapped call of the library refuses: test_call_arguments.py."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_2110_15362_b200 import binding as B
from paper_2110_15362_b200 import build

SOURCE = r"""
#include <stdint.h>
/* the widest call of the ABI: pointers, sizes, ints and one float among them; every argument into `seen` */
int all_of_them(const void *a, uint64_t b, int c, float t, void *d, void *e, void *f, uint64_t g, void *h, void *i, void *j,
                void *k, void *l, uint64_t m, void *n, uint64_t *seen, double *float_seen)
{
    uint64_t v[] = {(uint64_t)a, b, (uint64_t)(int64_t)c, (uint64_t)d, (uint64_t)e, (uint64_t)f, g, (uint64_t)h, (uint64_t)i,
                    (uint64_t)j, (uint64_t)k, (uint64_t)l, m, (uint64_t)n};
    for (int q = 0; q < 14; ++q) seen[q] = v[q];
    *float_seen = t;
    return -7;
}
int three(const void *a, uint32_t b, int c) { return a == 0 ? (int)b - c : 1000; }
"""


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    build.build_caller()
    from paper_2110_15362_b200 import _pycall
    d = tmp_path_factory.mktemp("pycall")
    (d / "f.c").write_text(SOURCE)
    subprocess.check_call(["gcc", "-O1", "-shared", "-fPIC", "-o", str(d / "f.so"), str(d / "f.c")])
    L = ctypes.CDLL(str(d / "f.so"))
    return lambda name: _pycall.native_call(ctypes.cast(getattr(L, name), ctypes.c_void_p).value)


@pytest.mark.parametrize("where", [0, 3, 9, 13])
def test_every_argument_arrives(call, where):
    """Tensors, buffers, None, large and negative integers and numpy integers in turn at every position."""
    t, buf = torch.zeros(4), (B.BatchItem * 2)()
    kinds = [(t, t.data_ptr()), (buf, ctypes.addressof(buf)), (None, 0), ((1 << 64) - 2, (1 << 64) - 2), (-3, (1 << 64) - 3),
             (np.int64(77), 77), (1 << 40, 1 << 40), (True, 1), (5, 5)]
    args = [kinds[(q + where) % len(kinds)] for q in range(14)]
    args[2] = (-9, (1 << 64) - 9)                                    # an int parameter
    seen, fseen = (ctypes.c_uint64 * 14)(), ctypes.c_double()
    fn = call("all_of_them")
    a = [v for v, _ in args]
    assert fn(*a[:3], 0.625, *a[3:], ctypes.addressof(seen), ctypes.addressof(fseen)) == -7
    assert list(seen) == [v for _, v in args]
    assert fseen.value == 0.625


def test_few_arguments_and_errors(call):
    fn = call("three")
    assert fn(None, 50, 8) == 42 and fn(torch.zeros(1), 50, 8) == 1000
    with pytest.raises(AttributeError):
        fn("text", 1, 2)
    with pytest.raises(TypeError):
        fn(*range(25))
    with pytest.raises(TypeError):
        fn(None, b=1)


def test_every_call_of_the_binding_is_wrapped():
    calls = B.lib().calls
    assert set(B.CALLS) <= set(B.EXPORTS) and "bt_compress" in B.CALLS
    for name in B.CALLS:
        assert callable(getattr(calls, name))
    A = 0x10000                                                      # a fake address: the call fails its checks first
    assert calls.bt_compress(A, 8192, 7, A, A, 8192, A, A, A, 1 << 20, A, None) == B.BT_ERR_DTYPE
    assert calls.bt_prune_fwd_compress(A + 4, 8192, B.BT_F32, 0.5, None, A, A, 8192, A, A, A, 1 << 20, A, None) == B.BT_ERR_ALIGN
