"""Densities where few particles reach a node (MIXED32): every node keeps the relative accuracy
of an FP64 sum, however small the weights that reach it, against exact rational arithmetic.
Particles lie far apart, two of them close to a periodic edge, with offsets near every place
where weights become small: 0, 1/2, 1, and tiny ones.

Bound, relative to the node's density: contributions are off by 2^-53 of themselves at most
(tests/test_density_weights.py); eight FP64 roundings at most follow or stand in their place:
those of a contribution formed in FP64, the conversion and scaling of the window's words, the
additions of the few blocks and particles that reach a node."""
from fractions import Fraction as Fr

import numpy as np
import pytest

import paper_1412_2480_gb300 as pic

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("tile", [0, 64])  # 64: nearly the largest window there is
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("order", [1, 2, 3])
def test_every_node_keeps_its_relative_accuracy(order, walls, tile):
    nx, ny = 160, 96
    rng = np.random.default_rng(order)
    k = np.arange(1, 25)
    near = np.concatenate((2.0 ** -k, 1.0 - 2.0 ** -k, 0.5 - 2.0 ** -(k + 1.0), 0.5 + 2.0 ** -k[1:], [0.0, 0.5, 2.0 ** -33,
                           2.0 ** -47 * 1.375], rng.random(30)))
    near = near.astype(np.float32).astype(np.float64)
    near = near[near < 1.0]
    cells = [(i, j) for j in range(0, ny, 6) for i in range(3 if walls else 0, nx - 6, 6)]
    parts = [(i, j, near[rng.integers(len(near))], near[rng.integers(len(near))]) for i, j in cells]
    # (a cell's index and a tiny offset fit one FP64 position only in cell 0)
    parts = [(i, j, a if i == 0 or a == 0 or a >= 2.0 ** -24 else 2.0 ** -24,
              b if j == 0 or b == 0 or b >= 2.0 ** -24 else 2.0 ** -24) for i, j, a, b in parts]
    x, y = np.array([p[0] + p[2] for p in parts]), np.array([p[1] + p[3] for p in parts])
    exact = {}
    for i, j, a, b in parts:
        bx, X = _weights(order, Fr(float(a)))
        by, Y = _weights(order, Fr(float(b)))
        for m, wy in enumerate(Y):
            for n, wx in enumerate(X):
                c = i + bx + n
                assert not walls or 0 <= c < nx
                key = ((j + by + m) % ny, c % nx)
                exact[key] = exact.get(key, 0) + wx * wy
    h = pic.pic_init(pic.pic_params_default(nx=nx, ny=ny, ppc=1, shape_order=order, gamma0=2.0, precision=pic.PIC_MIXED32,
                                            tile_x=tile, tile_y=tile,
                                            bc_x=pic.PIC_BC_WALLS if walls else pic.PIC_BC_PERIODIC))
    try:
        z = np.zeros(len(x))
        pic.pic_load_particles(h, 1, x, y, z, z, z)
        got = pic.fields_numpy(h, pic.PIC_DENSITY_E, nx, ny)
    finally:
        pic.pic_free(h)
    small = 0
    for kk in np.ndindex(ny, nx):
        want = exact.get(kk, Fr(0))
        assert abs(Fr(float(got[kk])) - want) <= want * 9 / 2 ** 53, (kk, got[kk], float(want))
        small += 0 < want < Fr(1, 2 ** 40)
    assert small > 0 or order == 1
