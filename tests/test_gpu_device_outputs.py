"""Quantities formed on demand into a caller's device array that no kernel may write as FP64:
one that starts between two multiples of 8 bytes. It goes through a copy and holds the same
bytes as an aligned array, and nothing beside it changes."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from runners import workload

pytestmark = pytest.mark.gpu


def _read(call, n, shift):
    import torch
    raw = torch.full((8 * n + 64,), 0x5A, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert call(raw.data_ptr() + 16 + shift) == pic.PIC_OK
    b = raw.cpu().numpy()
    body = slice(16 + shift, 16 + shift + 8 * n)
    assert np.all(np.delete(b, np.r_[body]) == 0x5A)
    return b[body].tobytes()


@pytest.mark.parametrize("precision", [pic.PIC_MIXED32, pic.PIC_FP64])
def test_device_arrays_of_any_alignment(precision):
    nx, ny, ppc = 40, 24, 3
    w, sp, F0 = workload(nx, ny, ppc, gamma0=3.0, u_th=0.3, seed=7, field_amp=0.05, colocated=False)
    h = pic.pic_init(pic.pic_params_default(nx=nx, ny=ny, ppc=ppc, gamma0=3.0, shape_order=2, precision=precision))
    try:
        for c in range(6):
            pic.pic_set_fields(h, c, np.ascontiguousarray(F0[c]).ravel())
        for s, d in enumerate(sp):
            pic.pic_load_particles(h, s, d["x"], d["y"], d["ux"], d["uy"], d["uz"])
        pic.pic_step(h, 1)
        L, n = pic.lib(), nx * ny
        for which in (pic.PIC_EX, pic.PIC_JX, pic.PIC_JX + 2):
            got = [_read(lambda p: L.pic_fields(h, which, p, n), n, shift) for shift in (0, 4, 1)]
            assert got[0] == got[1] == got[2]
        for which in (pic.PIC_RHO, pic.PIC_DENSITY_P, pic.PIC_DENSITY_E):  # (FP64 atomics: to rounding)
            a, b = (np.frombuffer(_read(lambda p: L.pic_fields(h, which, p, n), n, shift)) for shift in (0, 4))
            assert np.abs(a - b).max() <= 1e-13 * np.abs(a).max() + 1e-15
        m = pic.pic_particle_count(h, 0)
        a, b = (_read(lambda p: L.pic_particles(h, 0, p, m), 5 * m, shift) for shift in (0, 4))
        if precision == pic.PIC_FP64:
            assert a == b
    finally:
        pic.pic_free(h)
