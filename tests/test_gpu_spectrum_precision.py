"""The spectrum's rounding error against a sum in extended precision, over fixed seeds (the kernels
are deterministic, so the figure is one number per size). The limits are the error of a plain
FP64 Stockham transform, row by row and column by column, with every root rounded once
(1.67e-16 at 64 x 64, 1.80e-16 at 256 x 64, 2.23e-16 at 128 x 96, 3.42e-16 at 250 x 81), and
2% for the roots' last places: a form that rounds once more per value is 4 to 8% above it."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic

pytestmark = pytest.mark.gpu
L = np.longdouble


def _dft(n):
    k = (np.arange(n)[:, None] * np.arange(n)[None]) % n
    angle = -2 * np.arccos(L(-1)) * k.astype(L) / n
    return np.cos(angle), np.sin(angle)


@pytest.mark.parametrize("nx,ny,plain", [(64, 64, 1.674e-16), (256, 64, 1.796e-16), (128, 96, 2.228e-16), (250, 81, 3.420e-16)])
def test_error_of_noise(nx, ny, plain):
    (cx, sx), (cy, sy) = _dft(nx), _dft(ny)
    h = pic.pic_init(pic.pic_params_default(nx=nx, ny=ny, ppc=1, precision=pic.PIC_FP64))
    try:
        errors = []
        for seed in range(12):
            f = np.random.default_rng(seed).standard_normal((ny, nx))
            pic.pic_set_fields(h, pic.PIC_BZ, f.ravel())
            got = pic.pic_spectrum(h, pic.PIC_BZ, nx, ny).reshape(ny, nx).astype(L)
            re, im = f.astype(L) @ cx.T, f.astype(L) @ sx.T
            want = np.hypot(cy @ re - sy @ im, cy @ im + sy @ re) / (nx * ny)
            errors.append(float(((got - want) ** 2).sum() / (want ** 2).sum()))
    finally:
        pic.pic_free(h)
    assert np.sqrt(np.mean(errors)) <= 1.02 * plain
