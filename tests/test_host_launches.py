"""Host code of the C ABI over a fake device (tests/host_fake_runtime.cpp, host_fake_device.cu; no GPU): what a call
does when the runtime refuses a cooperative launch.  The launches per phase take over, every
step is taken once, and the handle keeps to them."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from inputs import generate as gen
from paper_1105_5613_gb300 import bbmd, build

HERE = os.path.dirname(os.path.abspath(__file__))


class Counts(C.Structure):
    _fields_ = [(k, C.c_int32) for k in ("begin", "grid_step", "grid_relax", "trigger_sort", "graph_launch",
                                         "sd_step", "force", "steps")]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake"))
    objs = []
    for src in (os.path.join(build.CSRC, "bbmd_api.cu"), os.path.join(HERE, "host_fake_device.cu")):
        obj = os.path.join(out, os.path.basename(src) + ".o")
        subprocess.run([build._nvcc(), *build.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-c", src, "-o", obj],
                       check=True)
        objs.append(obj)
    obj = os.path.join(out, "runtime.o")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-I", inc, "-c", os.path.join(HERE, "host_fake_runtime.cpp"), "-o", obj],
                   check=True)
    objs.append(obj)
    path = os.path.join(out, "libbbmd_fake.so")
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", path, *objs], check=True)
    L = C.CDLL(path)
    L.bbmd_create.argtypes = [C.POINTER(bbmd.bbmd_params), C.c_int64, C.POINTER(C.c_double), C.POINTER(C.c_uint8),
                              C.c_void_p, C.c_void_p, C.c_double, C.c_uint64, C.c_void_p, C.c_void_p,
                              C.POINTER(C.c_void_p)]
    L.bbmd_step.argtypes = [C.c_void_p, C.c_int64, C.c_double, C.c_void_p]
    L.bbmd_minimize.argtypes = [C.c_void_p, C.c_int64, C.c_double, C.c_double]
    L.bbmd_destroy.argtypes = [C.c_void_p]
    L.bbmd_step_launches.argtypes = [C.c_void_p]
    L.bbmd_step_launches.restype = C.c_int64
    return L


@pytest.fixture()
def handle(lib):
    made = []

    def make(ncell, shape):
        n = 4 * ncell ** 3
        box = np.full(3, gen.box_for(n, 1.2))
        sp = np.zeros(n, np.uint8)
        h = C.c_void_p()
        rc = lib.bbmd_create(C.byref(bbmd.ka_params(block_z=shape)), n, box.ctypes.data_as(C.POINTER(C.c_double)),
                             sp.ctypes.data_as(C.POINTER(C.c_uint8)), None, None, 1.0, 0, None, None, C.byref(h))
        assert rc == 0
        made.append(h)
        return h

    yield make
    lib.fake_reset(0, 0)
    for h in made:
        lib.bbmd_destroy(h)


def counts(lib):
    c = Counts()
    lib.fake_counts(C.byref(c))
    return c


@pytest.mark.parametrize("first", [0, 1, 2])
def test_steps_of_a_refused_launch_are_replayed(lib, handle, first):
    h = handle(10, 1)
    lib.fake_reset(1, first)  # the launches of 1024 steps after the first few are refused
    assert lib.bbmd_step(h, 2500, 0.005, None) == 0
    c = counts(lib)
    assert c.begin == 1 and c.steps == 2500 and c.grid_step == first + 1
    assert c.graph_launch == 2500 - 1024 * first
    assert lib.bbmd_step(h, 10, 0.005, None) == 0  # not tried again
    c = counts(lib)
    assert c.grid_step == first + 1 and c.steps == 2510


@pytest.mark.parametrize("first", [0, 1])
def test_descents_of_a_refused_launch_are_launched(lib, handle, first):
    h = handle(10, 1)
    lib.fake_reset(1, first)
    assert lib.bbmd_minimize(h, 1500, 1e-3, 0.05) == 0
    c = counts(lib)
    assert c.grid_relax == first + 1 and c.sd_step == 1500 - 1024 * first
    assert c.force == c.sd_step + 1  # each step's forces, and those of the last state
    assert lib.bbmd_minimize(h, 0, 1e-3, 0.05) == 0
    assert counts(lib).grid_relax == first + 1


@pytest.mark.parametrize("refuse", [2, 4, 8])
def test_a_refused_node_of_the_captured_step(lib, handle, refuse):
    h = handle(36, 1)  # past one wave of blocks: a captured step
    lib.fake_reset(refuse, 0)
    for total in (7, 12):
        assert lib.bbmd_step(h, 7 if total == 7 else 5, 0.005, None) == 0
        c = counts(lib)
        assert c.grid_step == 0 and c.graph_launch == total and c.trigger_sort == 1
    assert c.begin == 2


def test_nothing_refused(lib, handle):
    h, g = handle(10, 1), handle(36, 1)
    lib.fake_reset(0, 0)
    assert lib.bbmd_step(h, 1500, 0.005, None) == 0 and lib.bbmd_minimize(h, 30, 1e-3, 0.05) == 0
    c = counts(lib)
    assert (c.grid_step, c.grid_relax, c.graph_launch, c.steps) == (2, 1, 0, 1530)
    assert lib.bbmd_step(g, 9, 0.005, None) == 0
    assert counts(lib).graph_launch == 9 and counts(lib).trigger_sort == 1


def test_launches_are_counted(lib, handle):
    h, g = handle(10, 1), handle(36, 1)
    lib.fake_reset(0, 0)
    assert lib.bbmd_step_launches(h) == 0
    assert lib.bbmd_step(h, 2500, 0.005, None) == 0
    assert lib.bbmd_step_launches(h) == 1 + 3 + 2  # begin, launches of 1024, barriers cleared between
    assert lib.bbmd_step(h, 3, 0.002, None) == 0
    assert lib.bbmd_step_launches(h) == 6 + 2 + 1 + 1  # another dt: the pending update first
    assert lib.bbmd_step(g, 9, 0.005, None) == 0
    assert lib.bbmd_step_launches(g) == 1 + 9 * 6  # (the fake's graphs have six nodes)
    lib.fake_reset(1, 1)
    h = handle(10, 1)
    assert lib.bbmd_step(h, 1030, 0.005, None) == 0
    assert lib.bbmd_step_launches(h) == 1 + 1 + 1 + 6 * 6  # begin, 1024 steps, cleared, the rest replayed
