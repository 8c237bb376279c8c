"""Caps of the FP32 inner solves (csrc/inner_caps.h), host logic."""
import ctypes
import subprocess

import pytest

from tests.test_host_logic import CSRC


@pytest.fixture(scope="module")
def caps(tmp_path_factory):
    d = tmp_path_factory.mktemp("caps")
    src, so = d / "caps.cpp", d / "caps.so"
    src.write_text('#include "inner_caps.h"\n'
                   'extern "C" long long later(long long first, int early) {'
                   ' return nnqp::later_product_cap(first, early != 0); }\n'
                   'extern "C" long long first(long long n) { return nnqp::inner_product_cap(n); }\n')
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)])
    L = ctypes.CDLL(str(so))
    L.later.argtypes, L.later.restype = [ctypes.c_longlong, ctypes.c_int], ctypes.c_longlong
    L.first.argtypes, L.first.restype = [ctypes.c_longlong], ctypes.c_longlong
    return L


def test_room_of_the_later_solves_grows_with_the_first(caps):
    """At least 1,000 products and at least a quarter of the first solve's,
    never more than without the early ratios."""
    for n in (0, 1, 999, 1000, 2500, 4000, 4400, 5100, 20_000, 38_000, 100_000):
        base = max(n, 1000)
        assert caps.later(n, 0) == 2 * base
        assert caps.later(n, 1) - base >= max(1000, base // 4)
        assert caps.later(n, 1) <= caps.later(n, 0)
    assert caps.first(100) == 4000 and caps.first(1_000_000) == 64_000
