"""Shared-memory limits of the g(r) kernels over a fake of the runtime (no GPU): no call lowers
the limit that another thread's call, between its set and its launch, relies on, and no
launch asks for more than its kernel's limit.  Scratch is asked for where it is used."""
import ctypes as C
import os
import subprocess

import pytest

from paper_1105_5613_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("gr"))
    objs = []
    for src in (os.path.join(build.CSRC, "k_observe.cu"), os.path.join(HERE, "host_gr_launch.cu")):
        objs.append(os.path.join(out, os.path.basename(src) + ".o"))
        subprocess.run([build._nvcc(), *build.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-c", src, "-o", objs[-1]],
                       check=True)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    objs.append(os.path.join(out, "runtime.o"))
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-I", inc, "-c", os.path.join(HERE, "host_gr_runtime.cpp"), "-o",
                    objs[-1]], check=True)
    path = os.path.join(out, "libgr_fake.so")
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", path, *objs], check=True)
    L = C.CDLL(path)
    L.gr_call.argtypes = [C.c_double, C.c_int, C.c_int, C.c_double, C.c_int64]
    return L


def test_limits_are_never_lowered(lib):
    assert lib.gr_prepare() == 0
    out = (C.c_int * 3)()
    # over the build cells, on the coarse grid (too few build cells for rmax), all pairs
    for k, (L, nc, rmax) in enumerate([(40.0, 14, 3.0), (12.0, 3, 3.9), (12.0, 3, 5.0)]):
        for nbins in (4096, 1, 500, 4096, 2):
            assert lib.gr_call(L, nc, nbins, rmax, 1 << 20) == 0
        lib.fake_gr(out)
        assert out[0] == 0, "a limit was lowered"
        assert out[1] == 0, "a launch beyond its kernel's limit"
    assert out[2] == 5 + 5 * 5 + 5  # one kernel, five, one


def test_only_the_coarse_grid_takes_scratch(lib):
    assert lib.gr_prepare() == 0
    for nbins in (1, 500):
        assert lib.gr_call(40.0, 14, nbins, 3.0, 0) == 0  # over the build cells
        assert lib.gr_call(12.0, 3, nbins, 5.0, 0) == 0  # all pairs
        need = 2 * 1000 + 3 * (3 ** 3 + 1)
        assert lib.gr_call(12.0, 3, nbins, 3.9, need) == 0
        assert lib.gr_call(12.0, 3, nbins, 3.9, need - 1) == -1
