"""CPU: the edge table that the round kernel reads answers as the connections do."""
import os
import subprocess

import pytest

from paper_1912_00966_gb300 import build as libbuild

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("edge_table") / "edge_table")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", libbuild.INCLUDE, "-I", libbuild.CSRC,
                    "-I", os.path.join(libbuild.CUDA_HOME, "include"),
                    os.path.join(HERE, "c", "edge_table.cpp"),
                    os.path.join(libbuild.CSRC, "eat_build.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("stops,conns,t_max,dur_max,width,t0", [
    (1, 40, 500, 30, 60, 0),                 # one stop, every edge a loop
    (3, 400, 600, 90, 60, 0),                # several types and departures per slot: lists
    (3, 3000, 4000, 3, 3600, -5000),         # dense, nearly every departure undominated
    (40, 500, 90000, 1200, 3600, 0),         # sparse: most entries hold the next departure alone
    (5, 60, 400000, 100, 65535, 0),          # next departures beyond 16 bits
    (4, 200, 5000, 2**24 - 1, 600, 0),       # durations beyond 16 bits
    (2, 700, 50, 9, 1, 7),                   # one-second clusters
    (3, 30, 2**30, 500, 65535, -2**29),      # a span of decades, widest slots
    (600, 200000, 7000, 600, 600, 0),        # stops of more than 255 edges
])
@pytest.mark.parametrize("seed", [1, 2])
def test_edge_lookups(program, stops, conns, t_max, dur_max, width, t0, seed):
    r = subprocess.run([program, *map(str, (seed, stops, conns, t_max, dur_max, width, t0))],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
