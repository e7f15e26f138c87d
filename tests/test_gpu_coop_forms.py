"""The MIXED32 cooperative solve in its forms: tiles of 16, 32 and 64 rows (chosen by how many
tiles the grids have), quads of cells (every nx a multiple of 4) or single cells (any nx).
Each is compared with the WHILE-node solve of the same step (PIC_NO_COOP), which shares none
of its passes.

Bound: both stop at ||b - A x|| <= rtol ||b||, rtol = 1e-12, so their dB differ by at most
2e-12 kappa(A) (kappa < 3 at theta 1/2, CFL 1) in norm; E, B follow by one stencil of dB.
The current is an integer sum and equal to the bit."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from runners import rel, run_gpu, workload

pytestmark = pytest.mark.gpu


def _run(nx, ny, order, walls, flags, steps=1):
    w, sp, F0 = workload(nx, ny, 2, gamma0=3.0, u_th=0.3, seed=81, field_amp=0.05, colocated=False)
    if walls:
        F0 = F0.copy()
        F0[1:4, :, 0] = 0.0
    return run_gpu(nx, ny, 2, sp, F0, steps, order, gamma0=3.0, precision=pic.PIC_MIXED32, cg_rtol=1e-12, flags=flags,
                   bc_x=pic.PIC_BC_WALLS if walls else pic.PIC_BC_PERIODIC, want_particles=False)


@pytest.mark.parametrize("nx,ny,walls", [(8, 8, False), (9, 11, False), (13, 8, True), (64, 64, True), (66, 63, False),
                                         (127, 130, True), (512, 130, False), (511, 260, True), (1024, 333, False),
                                         (1021, 333, True)])
def test_solve_forms_agree_with_the_while_loop(nx, ny, walls):
    F, _, m = _run(nx, ny, 1, walls, 0)
    G, _, k = _run(nx, ny, 1, walls, pic.PIC_NO_COOP)
    assert 0 < m["cg_rel_resid"] <= 1e-12 and 0 < k["cg_rel_resid"] <= 1e-12
    np.testing.assert_array_equal(F[6:9], G[6:9])
    assert rel(F[9:12], G[9:12]) <= 6e-12
    assert rel(F[:6], G[:6]) <= 6e-12


def test_ragged_simulations_alone_and_in_a_batch_agree_bit_for_bit():
    sizes = [(33, 40), (50, 30), (64, 48), (130, 257)]
    mk = lambda nx, ny: pic.pic_params_default(nx=nx, ny=ny, ppc=2, gamma0=3.0, precision=pic.PIC_MIXED32, cg_rtol=1e-12)  # noqa: E731

    def load(h, k, nx, ny):
        _, sp, F0 = workload(nx, ny, 2, gamma0=3.0, u_th=0.3, seed=90 + k, field_amp=0.05, colocated=False)
        for c in range(6):
            pic.pic_set_fields(h, c, np.ascontiguousarray(F0[c]).ravel())
        for s, d in enumerate(sp):
            pic.pic_load_particles(h, s, d["x"], d["y"], d["ux"], d["uy"], d["uz"])

    def fields(h, nx, ny):
        return np.stack([pic.fields_numpy(h, c, nx, ny) for c in range(12)])

    h = pic.pic_init_batch([mk(*s) for s in sizes])
    try:
        for k, (nx, ny) in enumerate(sizes):
            pic.pic_select(h, k)
            load(h, k, nx, ny)
        pic.pic_step(h, 3)
        batch = []
        for k, (nx, ny) in enumerate(sizes):
            pic.pic_select(h, k)
            batch.append(fields(h, nx, ny))
    finally:
        pic.pic_free(h)
    for k, (nx, ny) in enumerate(sizes):
        h = pic.pic_init(mk(nx, ny))
        try:
            load(h, k, nx, ny)
            pic.pic_step(h, 3)
            np.testing.assert_array_equal(fields(h, nx, ny), batch[k])
        finally:
            pic.pic_free(h)
