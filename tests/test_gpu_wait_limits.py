"""The grid-wide waits of the FP64 PCG and of the MIXED32 solve on cells run out when their
bound is lowered to one poll: PIC_ETIMEOUT, nothing hangs, and with the default bound the same
handle meets its tolerance again. FP64 grids of each form of the kernel (one cell per thread,
two, vectors in memory), MIXED32 grids whose nx is no multiple of 4, alone and in a batch. A
solve in a single block waits for nobody."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from runners import workload

pytestmark = pytest.mark.gpu


def _handle(sizes, precision, **kw):
    prm = [pic.pic_params_default(nx=nx, ny=ny, ppc=1, gamma0=3.0, shape_order=1, precision=precision, cg_rtol=1e-10, **kw)
           for nx, ny in sizes]
    h = pic.pic_init_batch(prm)
    for k, (nx, ny) in enumerate(sizes):
        w, sp, F = workload(nx, ny, 1, gamma0=3.0, u_th=0.3, seed=51 + k, field_amp=0.05, colocated=False)
        pic.pic_select(h, k)
        for c in range(6):
            pic.pic_set_fields(h, c, np.ascontiguousarray(F[c]).ravel())
        for s, d in enumerate(sp):
            pic.pic_load_particles(h, s, d["x"], d["y"], d["ux"], d["uy"], d["uz"])
    pic.pic_select(h, 0)
    return h


@pytest.mark.parametrize("sizes,precision", [
    ([(128, 128)], pic.PIC_FP64), ([(512, 256)], pic.PIC_FP64), ([(512, 600)], pic.PIC_FP64),
    ([(258, 130)], pic.PIC_MIXED32), ([(97, 61), (130, 98)], pic.PIC_MIXED32)])
@pytest.mark.parametrize("graph", [True, False])
def test_waits_run_out_and_the_handle_goes_on(sizes, precision, graph):
    h = _handle(sizes, precision, flags=0 if graph else pic.PIC_NO_GRAPH)
    try:
        pic.pic_step(h, 1)
        assert 0 < pic.pic_moments(h)["cg_rel_resid"] <= 1e-10
        pic.pic_set_wait_limit(h, 1)
        with pytest.raises(pic.PicError) as e:
            pic.pic_step(h, 3)
        assert e.value.code == pic.PIC_ETIMEOUT, e.value
        assert pic.pic_moments(h)["step"] == 2  # the failing step completed, the rest were skipped
        pic.pic_set_wait_limit(h, 0)
        pic.pic_step(h, 2)
        for k in range(len(sizes)):
            pic.pic_select(h, k)
            m = pic.pic_moments(h)
            assert m["step"] == 4 and 0 < m["cg_rel_resid"] <= 1e-10
    finally:
        pic.pic_free(h)


def test_one_block_waits_for_nobody():
    h = _handle([(9, 9)], pic.PIC_MIXED32)  # (the FP64 PCG spreads 64 cells over two blocks)
    try:
        pic.pic_set_wait_limit(h, 1)
        pic.pic_step(h, 2)
        assert 0 < pic.pic_moments(h)["cg_rel_resid"] <= 1e-10
    finally:
        pic.pic_free(h)


@pytest.mark.parametrize("sizes,precision", [([(128, 128)], pic.PIC_FP64), ([(258, 130)], pic.PIC_MIXED32),
                                             ([(256, 128)], pic.PIC_MIXED32)])
def test_every_wait_that_runs_out_is_reported(sizes, precision):
    h = _handle(sizes, precision)
    try:
        pic.pic_set_wait_limit(h, 1)
        for k in range(3):
            with pytest.raises(pic.PicError) as e:
                pic.pic_step(h, 2)
            assert e.value.code == pic.PIC_ETIMEOUT, (k, e.value)
            assert pic.pic_moments(h)["step"] == k + 1
        pic.pic_set_wait_limit(h, 0)
        pic.pic_step(h, 2)
        assert 0 < pic.pic_moments(h)["cg_rel_resid"] <= 1e-10
    finally:
        pic.pic_free(h)
