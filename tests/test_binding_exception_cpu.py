"""A C++ exception that reaches the native part of the binding becomes a Python error, with the interpreter's lock held
again, and the module works on."""
import subprocess
import sys

from conftest import ROOT

STAND_IN = r'''
#include <stdexcept>
extern "C" int entry(const void*, void*, void*) { throw std::runtime_error("from the library"); }
'''
CHILD = r'''
import ctypes as C, sys
import torch
import paper_2110_15032_b200 as sbp
from paper_2110_15032_b200 import binding
from paper_2110_15032_b200 import _native
entry = C.cast(C.CDLL(sys.argv[1]).entry, C.c_void_p).value
_native.bind(*[entry] * len(binding._NATIVE_ENTRIES))

class Stream:
    cuda_stream = 0

t = sbp.SbpTensor((4,), torch.float32, sbp.B, [torch.zeros(4)])
for _ in range(3):
    try:
        _native.boxing(t, t, Stream())
        raise AssertionError("no error")
    except RuntimeError as e:
        assert "from the library" in str(e), e
print("held", sum(range(1000)))
'''


def test_an_exception_in_a_call_is_a_python_error(tmp_path):
    (tmp_path / "entry.cpp").write_text(STAND_IN)
    so = str(tmp_path / "entry.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-o", so, str(tmp_path / "entry.cpp")], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, so], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0 and "held 499500" in r.stdout, (r.returncode, r.stderr[-2000:])
