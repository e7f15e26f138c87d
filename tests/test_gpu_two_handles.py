"""A handle whose solve needs more shared memory than that of a handle made after it: simulations
by both inner solves in one handle (cg_rtol below 1e-13 keeps the CG) stage one partial sum per
chunk of cells. Both step, in either order."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from runners import workload

pytestmark = pytest.mark.gpu


def _handle(nx, ny):
    prm = [pic.pic_params_default(nx=a, ny=b, ppc=1, gamma0=3.0, shape_order=1, precision=pic.PIC_MIXED32, cg_rtol=rtol)
           for a, b, rtol in ((nx, ny, 1e-10), (32, 32, 1e-14))]
    h = pic.pic_init_batch(prm)
    w, sp, F = workload(32, 32, 1, gamma0=3.0, u_th=0.3, seed=81, field_amp=0.05, colocated=False)
    pic.pic_select(h, 1)
    for c in range(6):
        pic.pic_set_fields(h, c, np.ascontiguousarray(F[c]).ravel())
    for s, d in enumerate(sp):
        pic.pic_load_particles(h, s, d["x"], d["y"], d["ux"], d["uy"], d["uz"])
    return h


def test_a_later_handle_leaves_an_earlier_one_its_shared_memory():
    a = _handle(2048, 512)
    b = _handle(64, 64)
    try:
        for h in (a, b, a):
            pic.pic_step(h, 1)
            pic.pic_select(h, 1)
            assert 0 < pic.pic_moments(h)["cg_rel_resid"] <= 1e-14
    finally:
        pic.pic_free(a)
        pic.pic_free(b)
