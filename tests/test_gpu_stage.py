"""Positions at the edges of the load's rules: zero of either sign, the last number below the
box length, the length itself, outside the box by a little and by far, next to cell edges.
Positions in the box must come back as cell + FP32 offset of what went in, the others folded
first; both computed here with the same IEEE operations, so equality is exact."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic

pytestmark = pytest.mark.gpu


def _stored(x, n):
    L = float(n)
    x = x - np.floor(x / L) * L
    i = np.floor(x)
    f = (x - i).astype(np.float32)
    i, f = np.where(f >= 1, i + 1, i), np.where(f >= 1, np.float32(0), f)
    return i % n + f.astype(np.float64)


@pytest.mark.parametrize("nx,ny", [(40, 24), (8, 100)])
def test_positions_come_back_folded(nx, ny):
    def points(n):
        e = np.array([0.0, -0.0, 5e-324, 1e-30, np.nextafter(n, 0), float(n), np.nextafter(n, 2 * n), -1e-20, -0.25,
                      n + 3.75, 7.0 * n + 0.5, -3.0 * n - 0.125, 3.0, np.nextafter(3, 0), np.nextafter(3, 9), n - 1e-9,
                      n - 0.5])
        return np.concatenate([e, np.random.default_rng(n).uniform(0, n, 83)])
    x, y = points(nx), points(ny)[::-1].copy()
    h = pic.pic_init(pic.pic_params_default(nx=nx, ny=ny, ppc=2, gamma0=2.0, precision=pic.PIC_MIXED32))
    try:
        tag = np.arange(len(x), dtype=np.float64)
        pic.pic_load_particles(h, 0, x, y, tag, tag, tag)
        P = pic.pic_particles(h, 0)
    finally:
        pic.pic_free(h)
    P = P[:, np.argsort(P[2])]
    np.testing.assert_array_equal(P[0], _stored(x, nx))
    np.testing.assert_array_equal(P[1], _stored(y, ny))
