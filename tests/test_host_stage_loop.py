"""The order in which a CTA stages its blocks, compiled for the host over a model of the
mbarriers: kernels that run several bodies never initialise a live barrier, no buffer is
refilled while in use or in flight, and a wait that gives up is reported with no copy left
in flight.  Counts from a cell table that a launch left half sorted stay in range."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def loop(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("stage") / "host_stage_loop")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror",
                    os.path.join(HERE, "host_stage_loop.cpp"), "-o", exe], check=True)
    return lambda *a: subprocess.run([exe, *map(str, a)], check=True, capture_output=True,
                                     text=True).stdout.strip()


@pytest.mark.parametrize("buffers", [1, 2])
@pytest.mark.parametrize("blocks", [0, 1, 2, 4, 5, 8, 11, 20])
@pytest.mark.parametrize("bodies", [1, 2, 5])
def test_bodies_one_after_the_other(loop, buffers, blocks, bodies):
    assert loop(buffers, blocks, bodies, -1) == "ok"


@pytest.mark.parametrize("buffers", [1, 2])
@pytest.mark.parametrize("fail_at", [1, 4, 7, 19])
def test_a_wait_that_gives_up(loop, buffers, fail_at):
    assert loop(buffers, 20, 2, fail_at) == "ok"


def test_cells_of_a_table_half_sorted(loop):
    assert loop("cells") == "ok"
