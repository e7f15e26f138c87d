"""pic_spectrum in each of its forms, against numpy's FFT: transforms with every radix, rows
taken in pairs (an odd row left over), direct sums for other prime factors along either or
both axes, lengths around a direct block's edges, and the longest transform.

Bound, relative to the spectrum's largest amplitude: an N-point transform of data of RMS 1
carries rounding of about 1e-16 log2 N, a direct sum of N terms at most N 1e-16 = 4e-13 here
(the bound allows ten times the former and three times the latter)."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(8, 8), (9, 15), (11, 8), (8, 13), (25, 27), (128, 127), (257, 60), (510, 514),
                                   (1413, 247), (30, 2047), (2048, 9), (2049, 16), (2050, 11), (8192, 9), (9, 8192),
                                   (8200, 8), (4050, 11)])
def test_spectrum_forms(nx, ny):
    rng = np.random.default_rng(nx * 10007 + ny)
    f = rng.standard_normal((ny, nx)) + 3.0 * np.cos(2 * np.pi * (3 * np.arange(nx) / nx)[None, :])
    h = pic.pic_init(pic.pic_params_default(nx=nx, ny=ny))
    try:
        pic.pic_set_fields(h, pic.PIC_BZ, np.ascontiguousarray(f).ravel())
        got = pic.pic_spectrum(h, pic.PIC_BZ, nx, ny)
    finally:
        pic.pic_free(h)
    ref = np.abs(np.fft.fft2(f)) / (nx * ny)
    assert np.abs(got - ref).max() <= 1.2e-12 * ref.max()
