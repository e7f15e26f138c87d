"""Densities in whole numbers (MIXED32) against exact rational arithmetic: offsets at the edges
of every rule (zero, the smallest that the whole numbers hold and smaller ones, both sides of
1/2, the largest), cells at the edges of tiles and of the grid, and so many particles in one
place that a node's 64-bit sum wraps several times.

Bound: each contribution is within 8 units of 2^-56 of a full weight; the node's sum is then
rounded when it becomes FP64, when it is scaled and when up to 16 blocks add theirs: 32
roundings of 2^-53."""
from fractions import Fraction as Fr

import numpy as np
import pytest

import paper_1412_2480_gb300 as pic

pytestmark = pytest.mark.gpu
OFFSETS = [0.0, 2.0 ** -30, 2.0 ** -17, 2.0 ** -18 + 2.0 ** -41, 2.0 ** -10, 0.3, 0.5 - 2.0 ** -25, 0.5,
           0.5 + 2.0 ** -24, 0.8, 1.0 - 2.0 ** -24]


def _weights(order, f):
    if order == 1:
        return 0, [1 - f, f]
    if order == 2:
        up = f >= Fr(1, 2)
        d = f - 1 if up else f
        h = Fr(1, 2)
        return (0 if up else -1), [h * (h - d) ** 2, Fr(3, 4) - d * d, h * (h + d) ** 2]
    g = 1 - f
    return -1, [g ** 3 / 6, (4 - 6 * f ** 2 + 3 * f ** 3) / 6, (4 - 6 * g ** 2 + 3 * g ** 3) / 6, f ** 3 / 6]


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("walls", [False, True])
def test_density_is_exact_to_the_last_places(order, walls):
    nx, ny, tx, ty = 40, 24, 16, 8  # a ragged last tile in x
    f = np.float32(OFFSETS).astype(np.float64)
    cells = [(i, j) for i in (0, 5, 15, 16, 39) for j in (0, 7, 8, 23)]
    parts = [(i, j, a, b) for k, (i, j) in enumerate(cells) for m, a in enumerate(f) for b in f[(k + m) % 3::3]]
    parts += [(21, 11, 0.0, 0.0)] * 700 + [(33, 3, 0.5, f[5])] * 900
    x, y = np.array([p[0] + p[2] for p in parts]), np.array([p[1] + p[3] for p in parts])
    exact, count = {}, np.zeros((ny, nx))
    wt = {v: _weights(order, Fr(float(v))) for v in f}
    for i, j, a, b in parts:
        bx, X = wt[a]
        by, Y = wt[b]
        for m, wy in enumerate(Y):
            for n, wx in enumerate(X):
                c = i + bx + n
                if walls:
                    c = -c if c < 0 else 2 * nx - c if c > nx else c
                    if c == nx:
                        continue
                key = ((j + by + m) % ny, c % nx)
                exact[key] = exact.get(key, 0) + wx * wy
                count[key] += 1
    h = pic.pic_init(pic.pic_params_default(nx=nx, ny=ny, ppc=4, shape_order=order, gamma0=2.0, tile_x=tx, tile_y=ty,
                                            precision=pic.PIC_MIXED32,
                                            bc_x=pic.PIC_BC_WALLS if walls else pic.PIC_BC_PERIODIC))
    try:
        z = np.zeros(len(x))
        pic.pic_load_particles(h, 0, x, y, z, z, z)
        got = pic.fields_numpy(h, pic.PIC_DENSITY_P, nx, ny)
    finally:
        pic.pic_free(h)
    for k in np.ndindex(ny, nx):
        want = exact.get(k, Fr(0))
        bound = count[k] * 8 * 2.0 ** -56 + 32 * 2.0 ** -53 * float(want)
        assert abs(Fr(float(got[k])) - want) <= bound, (k, float(got[k]), float(want))
