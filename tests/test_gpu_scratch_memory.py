"""Large temporaries of read-backs and diagnostics go back to the device when the call returns,
and do not stay in the library's pool: particles of an FP64 handle (16 bytes each to the host)
and the spectrum of a large grid."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic

pytestmark = pytest.mark.gpu
KEPT = 80 << 20  # at most one temporary of 64 MB stays, and what the driver rounds it to


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_particles_of_an_fp64_handle():
    n = 12_000_000  # 192 MB of positions
    h = pic.pic_init(pic.pic_params_default(nx=64, ny=64, ppc=1, gamma0=2.0, precision=pic.PIC_FP64))
    try:
        x, z = np.full(n, 3.25), np.zeros(n)
        pic.pic_load_particles(h, 0, x, x, z, z, z)
        out = np.empty((5, n))
        before = _free()
        pic.pic_particles(h, 0, out)
        assert before - _free() <= KEPT
        assert np.all(out[:2] == 3.25) and np.all(out[2:] == 0.0)
    finally:
        pic.pic_free(h)


def test_spectrum_of_a_large_grid():
    nx, ny = 4096, 4096  # 134 MB each: the half spectrum, the amplitudes
    h = pic.pic_init(pic.pic_params_default(nx=nx, ny=ny, ppc=1, gamma0=2.0, precision=pic.PIC_FP64))
    try:
        F = np.cos(2 * np.pi * 3 * np.arange(nx) / nx)[None, :].repeat(ny, axis=0)
        pic.pic_set_fields(h, pic.PIC_BZ, F.ravel())
        before = _free()
        A = pic.pic_spectrum(h, pic.PIC_BZ, nx, ny)
        assert before - _free() <= KEPT
        assert abs(A.reshape(ny, nx)[0, 3] - 0.5) < 1e-12
    finally:
        pic.pic_free(h)
