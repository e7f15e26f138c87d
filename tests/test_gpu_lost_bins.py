"""A load whose particles all lie in one tile asks for bins that no device holds (MIXED32). The
load reports PIC_ENOMEM; the old bins are gone by then, so every later call that would run on
them says so instead of launching kernels on them, and the rest of the handle still answers."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic

pytestmark = pytest.mark.gpu


def test_calls_after_bins_could_not_be_allocated():
    nx, ny, n = 2048, 1024, 4_000_000  # 4096 tiles x 2 species x 5e6 slots x 24 bytes: about 1 TB
    h = pic.pic_init(pic.pic_params_default(nx=nx, ny=ny, ppc=1, gamma0=2.0, shape_order=1, precision=pic.PIC_MIXED32))
    try:
        z = np.zeros(n)
        few = [np.full(10, v) for v in (5.5, 7.25, 0.0, 0.0, 0.0)]
        for s in range(2):
            pic.pic_load_particles(h, s, *few)
        pic.pic_step(h, 1)
        with pytest.raises(pic.PicError) as e:
            pic.pic_load_particles(h, 0, np.full(n, 5.5), np.full(n, 7.25), z, z, z)
        assert e.value.code == pic.PIC_ENOMEM, e.value
        out = np.empty((5, 10))
        for call in (lambda: pic.pic_step(h, 1), lambda: pic.pic_profile(h, 1), lambda: pic.pic_conservation(h),
                     lambda: pic.fields_numpy(h, pic.PIC_RHO, nx, ny), lambda: pic.pic_particles(h, 1, out),
                     lambda: pic.pic_load_particles(h, 0, *few)):
            with pytest.raises(pic.PicError) as e:
                call()
            assert e.value.code == pic.PIC_ESTATE, e.value
            assert "lost" in str(e.value)
        assert np.all(np.isfinite(pic.fields_numpy(h, pic.PIC_EX, nx, ny)))
        assert pic.pic_moments(h)["step"] == 1
    finally:
        pic.pic_free(h)
    h = pic.pic_init(pic.pic_params_default(nx=32, ny=32, ppc=1, gamma0=2.0, precision=pic.PIC_MIXED32))
    try:
        for s in range(2):
            pic.pic_load_particles(h, s, *few)
        pic.pic_step(h, 2)
        assert abs(pic.fields_numpy(h, pic.PIC_DENSITY_P, 32, 32).sum() - 10) < 1e-12
    finally:
        pic.pic_free(h)
