"""The test that ends a grid-wide wait (csrc/arrivals.h), compiled for the host: right at every
count that can be seen, also where the 32-bit counter wraps, which a solve of a few million
iterations on 640 blocks reaches."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1412_2480_gb300", "csrc")


@pytest.fixture(scope="module")
def arrived(tmp_path_factory):
    d = tmp_path_factory.mktemp("arrivals")
    src, so = str(d / "a.cpp"), str(d / "a.so")
    with open(src, "w") as f:
        f.write('#include "arrivals.h"\nextern "C" int arrived(unsigned s, unsigned e, unsigned n) '
                "{ return pic::all_arrived(s, e, n); }\n")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    f = C.CDLL(so).arrived
    f.argtypes = [C.c_uint] * 3
    return f


@pytest.mark.parametrize("nblocks", [1, 2, 152, 608, 640])
def test_counter_may_wrap(arrived, nblocks):
    wrap = 2 ** 32 // nblocks
    for epoch in (1, 2, 1000, wrap - 1, wrap, wrap + 1, wrap + 2, 2 * wrap + 1, 2 ** 31 + 5):
        # counts seen while waiting for `epoch`: from one wait behind to one ahead
        for short in range(-nblocks, nblocks + 1):
            assert bool(arrived((epoch * nblocks + short) % 2 ** 32, epoch % 2 ** 32, nblocks)) == (short >= 0)
