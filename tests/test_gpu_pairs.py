"""The branch-free reciprocals, quotients and square roots of csrc/pairs.cuh
are correctly rounded over the ranges that their comment states: every float
of them for reciprocals, roots and constant divisors, 10^9 quotients."""
import ctypes as C
import os
import struct
import subprocess

import pytest
import torch

from paper_1809_06132_gb300 import _build

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("pairs") / "pairs_check.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "pairs_check.cu")
    subprocess.check_call([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-I" + _build.CSRC, "-shared", "-cudart", "static",
                           "-o", out, src])
    L = C.CDLL(out)
    for f in (L.check_unary, L.check_constant, L.check_quotients):
        f.restype = C.c_longlong
    L.check_unary.argtypes = [C.c_uint32, C.c_uint32, C.c_int]
    L.check_constant.argtypes = [C.c_uint32, C.c_uint32, C.c_float]
    L.check_quotients.argtypes = [C.c_int] * 4
    return L


def bits(x):
    return struct.unpack("<I", struct.pack("<f", x))[0]


FLT_MAX = struct.unpack("<f", struct.pack("<I", 0x7f7fffff))[0]


@pytest.mark.parametrize("roots,lo,hi", [(0, 2.0 ** -126, 2.0 ** 126), (1, 2.0 ** -100, FLT_MAX)])
def test_reciprocals_and_roots(lib, roots, lo, hi):
    assert lib.check_unary(bits(lo), bits(hi), roots) == 0


# window sizes, temperatures and a block's edge as the callers have them
@pytest.mark.parametrize("c", [25.0, 49.0, 81.0, 0.05, 0.3, 0.16, 0.8])
def test_constant_divisors(lib, c):
    assert lib.check_constant(bits(2.0 ** -100), bits(2.0 ** 120), c) == 0


# (variance products of a window reach down to 6e-14 = 2^-44)
@pytest.mark.parametrize("a0,a1,b0,b1", [(-60, 60, -60, 60), (-100, -60, -20, 20), (-60, 60, -60, -40), (-20, 0, -44, 10)])
def test_quotients(lib, a0, a1, b0, b1):
    assert lib.check_quotients(a0, a1, b0, b1) == 0
