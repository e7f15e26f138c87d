"""How tiles are cut into work items (csrc/tile_plan.h), compiled for the host: the size follows
from the particles there are, whatever room their bins have, and the parts cover what the bins
can hold. Also the sizes at which tests/test_gpu_tile_whole.py compares whole and split tiles."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1412_2480_gb300", "csrc")
SRC = """
#include "tile_plan.h"
extern "C" double size_of(double tiles, double resident, double mean) { return pic::split_size(tiles, resident, mean); }
extern "C" void split_of(double full, double mean, double size, int* out) {
    const pic::TileSplit t = pic::split_tile(full, mean, size);
    out[0] = t.parts;
    out[1] = t.pchunk;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = str(d / "p.cpp"), str(d / "p.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    L = C.CDLL(so)
    L.size_of.argtypes, L.size_of.restype = [C.c_double] * 3, C.c_double
    L.split_of.argtypes = [C.c_double] * 3 + [C.POINTER(C.c_int)]

    def split(tiles, resident, mean, full, own=None):  # own: the mean of the simulation's own tiles
        out = (C.c_int * 2)()
        L.split_of(full, own or mean, L.size_of(tiles, resident, mean), out)
        return out[0], out[1]
    return split


def _expect(ppc, tile=512):
    """The particles of a tile that a simulation is sized for (both species)."""
    return -(-(ppc * tile * 1.25 + 64) // 32) * 32 * 1.6


@pytest.mark.parametrize("tiles,resident,ppc,parts", [(8, 456, 8, 32), (32, 456, 100, 14), (2048, 456, 32, 1)])
def test_known_splits(plan, tiles, resident, ppc, parts):
    n = _expect(ppc)
    got = plan(tiles, resident, n, n)
    assert got[0] == parts
    assert 0 <= got[0] * got[1] - n < 256 * parts + 256  # every part has work, and all of them hold the tile


@pytest.mark.parametrize("tiles,resident,ppc", [(8, 456, 8), (32, 304, 100), (720, 456, 50), (2048, 608, 32)])
def test_room_in_the_bins_does_not_change_the_size(plan, tiles, resident, ppc):
    n = _expect(ppc)
    parts, chunk = plan(tiles, resident, n, n)
    for room in (2.0, 4.0, 40.0):
        p, c = plan(tiles, resident, n, room * n)
        assert c == chunk and parts <= p <= parts + n / 1000 + 1
    assert plan(tiles, resident, n, n / 4)[1] == chunk  # (bins smaller than the particles: shares grow at run time)


def test_few_particles_in_large_bins(plan):
    parts, chunk = plan(4096, 456, 0.5, 1e6)
    assert chunk == 256 and parts == 1  # (they would cost more than they hold)
    assert plan(2048, 456, 8000, 2e5)[0] == 9


@pytest.mark.parametrize("resident", [152, 304, 456, 608, 912])
def test_whole_and_split_in_the_gpu_test(plan, resident):
    # 2048 x 1024 cells beside it: 4096 tiles of 32 x 16
    for tiles, cells in ((8, 512), (9, 512)):
        n = _expect(12, cells)
        assert plan(tiles, resident, n, n)[0] > 1                                   # alone
        mean = (n * tiles + _expect(12) * 4096) / (tiles + 4096)
        assert plan(tiles + 4096, resident, mean, n, n)[0] == 1                        # beside it
