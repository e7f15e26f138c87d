"""Densities and momentum from each place a particle can be (MIXED32), and it is known which:
outboxes after a step without a re-sort, and the overflow list after a step that ended before
its re-sort (the solve is allowed one iteration). Against sums in FP64 over the particles that
pic_particles returns.

Bound: positions come back exactly (a cell and an FP32 offset in one FP64 number, to 2^-46);
a node is a sum of up to 400 terms of relative error 2^-52 on either side, and a term's
weights move by 2^-45 with its position: 1e-13 of the largest density."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from runners import workload
from test_gpu_density import _density

pytestmark = pytest.mark.gpu


def _check(h, nx, ny, order, walls):
    P = [pic.pic_particles(h, s) for s in range(2)]
    mw = pic.pic_moments(h)["macro_weight"]
    rho = [pic.fields_numpy(h, which, nx, ny) for which in (pic.PIC_DENSITY_P, pic.PIC_DENSITY_E)]
    both = pic.fields_numpy(h, pic.PIC_RHO, nx, ny)
    cons = pic.pic_conservation(h)
    for got, p in zip(rho, P):
        ref = _density(p, nx, ny, order, walls)
        assert np.abs(got - ref).max() <= 1e-13 * ref.max()
    assert np.abs(both - mw * (rho[0] - rho[1])).max() <= 1e-13 * mw * rho[0].max()
    mom = mw * sum(p[2:].sum(axis=1) for p in P)
    np.testing.assert_allclose(cons["momentum"], mom, rtol=0, atol=1e-12 * mw * np.abs(P[0][2:]).sum())


@pytest.mark.parametrize("order,walls", [(1, False), (2, False), (2, True), (3, False), (3, True)])
def test_outboxes_and_overflow_list(order, walls):
    nx, ny, ppc = 72, 40, 20
    w, sp, F0 = workload(nx, ny, ppc, gamma0=3.0, u_th=0.5, seed=92, field_amp=0.02, colocated=False)
    if walls:
        F0 = F0.copy()
        F0[1:4, :, 0] = 0.0
    for declared, max_iter in ((ppc, 200), (1, 1)):
        h = pic.pic_init(pic.pic_params_default(nx=nx, ny=ny, ppc=declared, gamma0=3.0, shape_order=order, cg_rtol=1e-10,
                                                cg_max_iter=max_iter, precision=pic.PIC_MIXED32,
                                                bc_x=pic.PIC_BC_WALLS if walls else pic.PIC_BC_PERIODIC))
        try:
            for c in range(6):
                pic.pic_set_fields(h, c, np.ascontiguousarray(F0[c]).ravel())
            for s, d in enumerate(sp):
                pic.pic_load_particles(h, s, d["x"], d["y"], d["ux"], d["uy"], d["uz"])
            before = pic.pic_moments(h)
            if declared == ppc:
                pic.pic_step(h, 1)
            else:
                with pytest.raises(pic.PicError) as e:
                    pic.pic_step(h, 1)
                assert e.value.code == pic.PIC_ECG_NOCONV, e.value
            after = pic.pic_moments(h)
            assert after["rebins"] == before["rebins"]  # the particles are where the step left them
            parked = after["overflow_moves"] - before["overflow_moves"]
            assert parked == 0 if declared == ppc else parked > 100
            _check(h, nx, ny, order, walls)
        finally:
            pic.pic_free(h)
