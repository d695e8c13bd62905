"""The colours in which the adjoints' band solve updates its nodes in place
(paper_1503_08406_gb300/csrc/lbm_flow_adjoint.cuh), built for the host: no two
neighbours share one, on walled and periodic y axes of any length, and the list
holds each colour's nodes in a range of their own."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1503_08406_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("band") / "libband.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", out,
                    os.path.join(HERE, "native", "band_order_host.cpp")], check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("per_y", [0, 1])
@pytest.mark.parametrize("percent", [0, 30, 100])
def test_no_neighbours_of_one_colour(lib, per_y, percent):
    for nx in (3, 4, 5, 40, 41):
        for ny in range(3, 40):
            got = lib.band_order_check(nx, ny, per_y, percent, nx + ny)
            assert got == 0, (nx, ny, got)
