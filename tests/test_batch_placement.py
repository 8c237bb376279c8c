"""Placement of the instances of a batched solve (csrc/batch_place.h), host
logic only: every instance gets a place that the device schedules and whose
shared memory fits, whatever sizes of clusters the device refuses."""
import ctypes
import subprocess

import pytest

from tests.test_host_logic import CSRC

SMEM = 204 * 1024


@pytest.fixture(scope="module")
def place(tmp_path_factory):
    d = tmp_path_factory.mktemp("place")
    src = d / "place.cpp"
    src.write_text(
        '#include "batch_place.h"\n'
        'using namespace nnqp;\n'
        '// bits c of local / memory: clusters of c CTAs are scheduled\n'
        'extern "C" int place(long long slices, long long widest, int vbytes, long long target, int most, int local,\n'
        '                     int memory, int *is_local) {\n'
        '    ResPlace p = place_instance(slices, widest, vbytes, target, most,\n'
        '                                [&](int c, bool l) { return ((l ? local : memory) >> c & 1) != 0; });\n'
        '    *is_local = p.local; return p.cluster; }\n'
        'extern "C" int plain(int most, int can) { return plain_cluster(most, [&](int c) { return (can >> c & 1) != 0; }); }\n'
        'extern "C" long long bytes(long long per, long long slots, int vbytes) {\n'
        '    return (long long)batch_res_bytes(per, slots, vbytes); }\n')
    so = d / "place.so"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)])
    L = ctypes.CDLL(str(so))
    L.place.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_longlong, ctypes.c_int,
                        ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    L.bytes.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int]
    L.bytes.restype = ctypes.c_longlong
    return L


def up_to(c):
    return sum(1 << k for k in (1, 2, 4, 8, 16) if k <= c)


def at(L, slices, widest, vbytes, target, most=16, local=up_to(16), memory=up_to(16)):
    q = ctypes.c_int()
    c = L.place(slices, widest, vbytes, target, most, local, memory, ctypes.byref(q))
    return c, bool(q.value)


def test_a_device_that_schedules_all_sizes(place):
    """As few CTAs as give each at most the target, or as many as the operator
    needs; the operator outside where even 16 do not hold it."""
    assert at(place, 12, 192, 8, 24) == (1, True)
    assert at(place, 25, 192, 8, 24) == (2, True)
    assert at(place, 444, 192, 8, 24) == (16, True)
    assert at(place, 444, 192, 8, 24, most=8) == (8, False)
    assert at(place, 1000, 192, 8, 24) == (16, False)
    assert at(place, 4000, 192, 8, 24) == (0, False)
    assert at(place, 40, 2048, 8, 24) == (8, True)       # 24 slices of 64-entry rows do not fit


@pytest.mark.parametrize("most", [0, 1, 2, 4, 8, 16])
@pytest.mark.parametrize("vbytes", [4, 8])
@pytest.mark.parametrize("target", [4, 11, 24])
def test_refused_sizes_leave_a_place_that_exists(place, most, vbytes, target):
    for slices in (1, 5, 30, 100, 443, 700, 2000, 20000):
        for widest in (64, 192, 448, 2048):
            for memory in (up_to(most), 0):
                c, local = at(place, slices, widest, vbytes, target, local=up_to(most), memory=memory)
                if c == 0:
                    assert most == 0 or place.bytes(-(-slices // most), widest, vbytes) > SMEM
                    continue
                assert c <= most and (local or memory >> c & 1)
                assert place.bytes(-(-slices // c), widest if local else 0, vbytes) <= SMEM
                # never refused a size that the full device's place takes
                if at(place, slices, widest, vbytes, target)[0] <= most and local:
                    assert (c, local) == at(place, slices, widest, vbytes, target)
    assert place.plain(16, up_to(most)) == max(most, 1)
