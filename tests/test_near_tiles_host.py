"""The tiles that a split step leaves for its near-tile pass
(paper_1503_08406_gb300/csrc/lbm_tiles.cuh), built for the host: whatever node a
listed tile's enthalpy region holds lies in a near tile, whichever way the region
wraps, and the units of the near-tile pass take every part of a near tile once."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1503_08406_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("near") / "libnear.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", out,
                    os.path.join(HERE, "native", "near_tiles_host.cpp")], check=True)
    return ctypes.CDLL(out)


# the other axis: one tile, three, and five with a last one 3 nodes wide
@pytest.mark.parametrize("other", [12, 96, 131])
@pytest.mark.parametrize("per", [(0, 0), (1, 0), (0, 1), (1, 1)])
def test_near_tiles_hold_every_region(lib, per, other):
    for n in range(3, 227):
        for nx, ny in ((n, other), (other, n)):
            for seed, (count, cross) in enumerate(((1, 0), (1, 0), (3, 0), (1, 1), (9, 1))):
                got = lib.near_tiles_check(nx, ny, per[0], per[1], count, cross, 10 * n + seed)
                assert got == 0, (nx, ny, per, count, cross, seed, got)


@pytest.mark.parametrize("nx,ny", [(129, 100), (100, 129), (129, 131), (128, 99)])
def test_each_single_tile(lib, nx, ny):
    for seed in range(200):
        assert lib.near_tiles_check(nx, ny, 1, 1, 1, 0, seed) == 0, seed


def test_mapped_lattice(lib):
    """More than 1152 tiles: the near map, and the near pass from the list."""
    for nx, ny in ((36865, 131), (4097, 1029), (4096, 1024)):
        for count in (1, 40):
            assert lib.near_tiles_check(nx, ny, 1, 1, count, 0, count) == 0
