"""The density's contributions in whole numbers (csrc/density_fixed.h), compiled for the host,
against exact rational arithmetic: each keeps its relative accuracy however small it is, a
particle that would lose it is refused, and none that has no small contribution is.

Bounds: at order 1 contributions are exact; at order 2 each is cut off below 2^-88, or is a
difference of two that are, and at least 2^-34: 2^-53; at order 3 products of factors that are
off by 2^-57, cut off below 2^-88 where they are 2^-35 or more: 2^-53 again. The smallest words
are those of a sum: the highest is 2^24 at most, which is what a window's 2^32 are counted by."""
import ctypes as C
import os
import random
import struct
import subprocess
from fractions import Fraction as Fr

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1412_2480_gb300", "csrc")
SRC = """
#include "density_fixed.h"
using namespace pic;
template <int P> int run(unsigned bx, unsigned by, int* first, unsigned* out) {
    unsigned Fx, Fy;
    if (!(fixed_offset(bx, Fx) & fixed_offset(by, Fy))) return -1;
    for (int k = 0; k < 48; k++) out[k] = 0;
    first[0] = first[1] = 1000;
    const bool ok = density_contributions<P>(10, Fx, 20, Fy, [&](int i, int by, int r, const Words (&v)[P + 1]) {
        const int j = by + r;
        first[0] = i;
        if (j < first[1]) first[1] = j;
        for (int a = 0; a <= P; a++)
            for (int k = 0; k < 3; k++) out[((j - 19) * 4 + a) * 3 + k] = v[a].w[k];  // rows 19..22
    });
    return ok ? 1 : 0;
}
extern "C" int contributions(int order, unsigned bx, unsigned by, int* first, unsigned* out) {
    return order == 1 ? run<1>(bx, by, first, out) : order == 2 ? run<2>(bx, by, first, out) : run<3>(bx, by, first, out);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("density")
    src, so = str(d / "d.cpp"), str(d / "d.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Wno-unknown-pragmas", "-shared", "-fPIC", "-I", CSRC, src, "-o", so],
                   check=True)
    return C.CDLL(so)


def _exact(order, f):
    if order == 1:
        return 0, [1 - f, f]
    if order == 2:
        up = f >= Fr(1, 2)
        d = f - 1 if up else f
        h = Fr(1, 2)
        return (0 if up else -1), [h * (h - d) ** 2, Fr(3, 4) - d * d, h * (h + d) ** 2]
    g = 1 - f
    return -1, [g ** 3 / 6, (4 - 6 * f ** 2 + 3 * f ** 3) / 6, (4 - 6 * g ** 2 + 3 * g ** 3) / 6, f ** 3 / 6]


def _value(bits):
    return Fr(struct.unpack("<f", struct.pack("<I", bits))[0])


def _offsets():
    rng = random.Random(4)
    bits = [0, 1, 0x00800000, 0x3f7fffff, 0x3f000000, 0x3effffff, 0x3f000001, 0x3e800000]
    bits += [(127 - k) << 23 for k in range(1, 40)]                         # powers of two
    bits += [((127 - k) << 23) + rng.randrange(1 << 23) for k in range(1, 40)]
    for k in range(1, 24):                                                   # close to 1 and to 1/2
        bits += [0x3f800000 - (1 << k), 0x3f800000 - rng.randrange(1, 1 << k), 0x3f000000 + (1 << (k - 1)) - 1,
                 0x3f000000 - rng.randrange(1, 1 << k), 0x3f000000 + rng.randrange(1 << (k - 1))]
    bits += [struct.unpack("<I", struct.pack("<f", rng.random() * (1 - 2 ** -24)))[0] for _ in range(300)]
    return [b for b in bits if b < 0x3f800000]


@pytest.mark.parametrize("order", [1, 2, 3])
def test_contributions(lib, order):
    rng = random.Random(order)
    unit = {1: Fr(1, 2 ** 62), 2: Fr(1, 2 ** 88), 3: Fr(4, 9) / 2 ** 88}[order]
    offs = _offsets()
    first, out = (C.c_int * 2)(), (C.c_uint * 48)()
    taken = 0
    for _ in range(6000):
        x, y = rng.choice(offs), rng.choice(offs)
        rc = lib.contributions(order, C.c_uint(x), C.c_uint(y), first, out)
        fx, fy = _value(x), _value(y)
        whole = all((f * 2 ** 31).denominator == 1 and (f == 0 or f >= Fr(1, 256)) for f in (fx, fy))
        assert (rc >= 0) == whole
        if rc < 0:
            continue
        (bx, wx), (by, wy) = _exact(order, fx), _exact(order, fy)
        want = {(a, b): u * v for a, u in enumerate(wx) for b, v in enumerate(wy)}
        least = min(v for v in want.values() if v)
        assert rc == 1 or (order > 1 and least < Fr(1, 2 ** 29))
        if rc == 0:
            continue
        taken += 1
        assert least > Fr(1, 2 ** 38) or order == 1
        assert (first[0], first[1]) == (10 + bx, 20 + by)
        total = 0
        for (a, b), w in want.items():
            o = ((first[1] - 19 + b) * 4 + a) * 3
            v = (out[o + 2] << 64) + (out[o + 1] << 32) + out[o]
            assert out[o + 2] <= 1 << 24
            total += v
            assert abs(unit * v - w) <= (0 if order == 1 else w / 2 ** 53), (order, hex(x), hex(y), a, b, float(unit * v), float(w))
        assert order == 3 or unit * total == 1
    assert taken > 500
