"""Work units of large plans (csrc/units.h): every point of every replication lies in exactly one unit
and the unit count stays below 2^32 over the whole accepted range, N <= 2^31 and M <= 65535.  Host
arithmetic alone; a plan of these sizes is never built here."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1408_5526_gb300", "csrc")


class Shape(C.Structure):
    _fields_ = [("ppt", C.c_int), ("tile", C.c_uint32), ("tiles_per_m", C.c_uint32), ("units", C.c_uint32)]


@pytest.fixture(scope="module")
def shape(tmp_path_factory):
    d = tmp_path_factory.mktemp("units")
    src, lib = d / "u.cpp", d / "u.so"
    src.write_text('#include "units.h"\nextern "C" void shape(uint64_t N, uint32_t M, int t, int p, '
                   'rqmc::UnitShape *s) { *s = rqmc::unit_shape(N, M, t, p); }\n')
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    f = C.CDLL(str(lib)).shape
    f.argtypes = [C.c_uint64, C.c_uint32, C.c_int, C.c_int, C.POINTER(Shape)]
    f.restype = None

    def call(N, M, threads, ppt):
        s = Shape()
        f(N, M, threads, ppt, C.byref(s))
        return s

    return call


@pytest.mark.parametrize("threads, ppt", [(64, 1), (64, 2), (128, 1), (256, 2), (32, 8), (256, 64)])
@pytest.mark.parametrize("N, M", [(1, 1), (1, 65535), (4097, 31), (1 << 31, 1), (1 << 31, 127), (1 << 31, 128),
                                  (1 << 31, 256), (1 << 31, 300), ((1 << 31) - 1, 2048), (1 << 31, 65535)])
def test_units_cover_every_point_in_32_bits(shape, N, M, threads, ppt):
    s = shape(N, M, threads, ppt)
    assert s.units < (1 << 32) - 1 and s.units == s.tiles_per_m * M
    assert s.tile == threads * s.ppt and s.ppt % ppt == 0
    assert (s.tiles_per_m - 1) * s.tile < N <= s.tiles_per_m * s.tile < 1 << 32
    if -(-N // (threads * ppt)) * M < (1 << 32) - 1:   # the usual tile wherever its count fits
        assert s.ppt == ppt
