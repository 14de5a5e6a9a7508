"""CPU: the edge table on uneven timetables, and without threads or memory to build it."""
import os
import subprocess

import pytest

from paper_1912_00966_gb300 import build as libbuild

HERE = os.path.dirname(os.path.abspath(__file__))


def _compiled(folder, name):
    exe = str(folder / name)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", libbuild.INCLUDE, "-I", libbuild.CSRC,
                    "-I", os.path.join(libbuild.CUDA_HOME, "include"),
                    os.path.join(HERE, "c", name + ".cpp"),
                    os.path.join(libbuild.CSRC, "eat_build.cpp"), "-o", exe, "-ldl"], check=True)
    return exe


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    return _compiled(tmp_path_factory.mktemp("edge_lists"), "edge_lists")


@pytest.mark.parametrize("stops,rare,headway,days,extra", [
    (300, 2000, 60, 1, 0),        # a metro among edges of a few departures a day
    (900, 9000, 5, 1, 0),         # one every five seconds: parts of parts
    (4, 0, 600, 1, 400),          # a single departure a year on makes the slots their longest
    (200, 300, 1, 1, 60),         # every second, widest slots: three levels
    (50, 50, 30, 5, 0),           # days without end, most entries empty
    (4, 0, 2, 1, 0),              # slots as short as they come: no table
])
@pytest.mark.parametrize("seed", [1, 2])
def test_busy_edges(program, stops, rare, headway, days, extra, seed):
    """Every lookup equals the connections' and takes seven loads at most; walked from its start, a
    list of the busy edges took up to thousands."""
    r = subprocess.run([program, *map(str, (seed, stops, rare, headway, days, extra))],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


def test_built_without_threads_or_memory(tmp_path):
    """A thread that cannot be started is done without, an allocation that fails is EAT_ERR_OOM."""
    r = subprocess.run([_compiled(tmp_path, "edge_limits")], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout + r.stderr)
