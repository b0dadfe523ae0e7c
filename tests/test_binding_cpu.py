"""The native part of the binding describes a tensor as the ctypes descriptor does.

The module is bound, in a process of its own, to a stand-in whose boxing entry point keeps a copy of the
two descriptors it is handed, so nothing of the library runs and no GPU is needed."""
import subprocess
import sys

from conftest import ROOT

CHILD = r'''
import ctypes as C
import torch
import paper_2110_15032_b200 as sbp
from paper_2110_15032_b200 import binding
from paper_2110_15032_b200.build import build
build()
from paper_2110_15032_b200 import _native

kept = []
PROTO = C.CFUNCTYPE(C.c_int, C.POINTER(binding._Tensor), C.POINTER(binding._Tensor), C.c_void_p)

@PROTO
def boxing(a, b, stream):
    kept.append((C.string_at(a, C.sizeof(binding._Tensor)), C.string_at(b, C.sizeof(binding._Tensor)), stream))
    return 0

addr = C.cast(boxing, C.c_void_p).value
_native.bind(*[addr] * len(binding._NATIVE_ENTRIES))

class Stream:
    cuda_stream = 0x1234

def same(a, b):
    kept.clear()
    assert _native.boxing(a, b, Stream()) == 0
    assert kept[0] == (bytes(a._c()), bytes(b._c()), 0x1234), (a.shape, a.sig)

def host(shape, dtype, sig, k):
    p = tuple(k) if isinstance(k, tuple) else None
    n = k if p is None else p[0] * p[1]
    return sbp.SbpTensor(shape, dtype, sig, [torch.zeros(sbp.sbp_local_shape(shape, sig, k, r, dtype), dtype=dtype) for r in range(n)], p)

for dtype in (torch.float32, torch.bfloat16, torch.int64):
    same(host((7, 5), dtype, sbp.S(0), 3), host((7, 5), dtype, sbp.B, 16))
    same(host((2, 3, 4, 5), dtype, sbp.S(3), 2), host((9,), dtype, sbp.P_MAX, 1))
    same(host((8, 6), dtype, (sbp.S(0), sbp.P_SUM), (2, 3)), host((8, 6), dtype, (sbp.B, sbp.S(1)), (2, 3)))
big = torch.zeros(10, 12)
window = sbp.SbpTensor((10, 8), torch.float32, sbp.S(1), [big[:, :4], big[:, 4:8]])
same(window, sbp.SbpTensor((8, 8), torch.float32, sbp.B, [None, torch.zeros(8, 8)]))
same(sbp.SbpTensor((0, 8), torch.float32, sbp.S(0), [torch.zeros(0, 8)] * 2), host((8,), torch.int64, sbp.B, 2))

def refused(exc, *a):
    try:
        _native.boxing(*a)
    except exc:
        return
    raise AssertionError((exc, a))

ok = host((8, 6), torch.float32, sbp.B, 2)
bad = host((8, 6), torch.float32, sbp.B, 2)
bad.locals[1] = torch.zeros(8, 12)[:, ::2]
refused(ValueError, ok, bad, Stream())
bad.locals[1] = 3
refused(TypeError, ok, bad, Stream())
wide = host((8, 6), torch.float32, sbp.B, 2)
wide.locals = [torch.zeros(8, 6)] * 17
refused(IndexError, ok, wide, Stream())
other = host((8, 6), torch.float32, sbp.B, 2)
other.dtype = torch.float16
refused(KeyError, ok, other, Stream())
refused(AttributeError, ok, 5, Stream())
refused(AttributeError, ok, ok, 5)
refused(TypeError, ok, ok)
print("ok")
'''


def test_native_descriptors_equal_the_ctypes_ones():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
