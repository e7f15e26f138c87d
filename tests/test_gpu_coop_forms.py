"""The MIXED32 cooperative solve in its forms: tiles of 16, 32 and 64 rows (chosen by how many
tiles the grids have), for grids whose nx is a multiple of 4; cell by cell for any other nx.
Each is compared with the WHILE-node solve of the same step (PIC_NO_COOP). The form on tiles
shares none of its passes; the one on cells runs the same arithmetic and sums in the same
order, and must give the same bits over several steps, alone and in a batch.

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


def _fields(sizes, flags, walls=False, steps=5):
    """Fields after some steps of a batch of simulations (or one)."""
    mk = lambda nx, ny: pic.pic_params_default(nx=nx, ny=ny, ppc=2, gamma0=3.0, precision=pic.PIC_MIXED32, flags=flags,  # noqa: E731
                                               bc_x=pic.PIC_BC_WALLS if walls else pic.PIC_BC_PERIODIC)
    h = pic.pic_init_batch([mk(*s) for s in sizes])
    try:
        out = []
        for k, (nx, ny) in enumerate(sizes):
            pic.pic_select(h, k)
            _, sp, F0 = workload(nx, ny, 2, gamma0=3.0, u_th=0.3, seed=90 + nx, field_amp=0.05, colocated=False)
            if walls:
                F0 = F0.copy()
                F0[1:4, :, 0] = 0.0
            for c in range(6):
                pic.pic_set_fields(h, c, np.ascontiguousarray(F0[c]).ravel())
            for s, d in enumerate(sp):
                pic.pic_load_particles(h, s, d["x"], d["y"], d["ux"], d["uy"], d["uz"])
        pic.pic_step(h, steps)
        for k, (nx, ny) in enumerate(sizes):
            pic.pic_select(h, k)
            out.append(np.stack([pic.fields_numpy(h, c, nx, ny) for c in range(12)]))
        return out
    finally:
        pic.pic_free(h)


@pytest.mark.parametrize("sizes,walls", [
    ([(9, 11)], False), ([(13, 40)], True), ([(255, 8)], False), ([(257, 129)], True), ([(1413, 247)], False),
    ([(33, 40), (50, 30), (64, 48), (130, 257)], False), ([(64, 48), (33, 40)], True)])
def test_ragged_grids_give_the_while_loops_bits(sizes, walls):
    for a, b in zip(_fields(sizes, 0, walls), _fields(sizes, pic.PIC_NO_COOP, walls)):
        np.testing.assert_array_equal(a, b)


def test_ragged_simulations_alone_and_in_a_batch_agree_bit_for_bit():
    # (each ragged: one whose nx is a multiple of 4 takes the form on tiles when alone)
    sizes = [(33, 40), (50, 30), (62, 48), (130, 257)]
    for s, b in zip(sizes, _fields(sizes, 0, steps=3)):
        np.testing.assert_array_equal(_fields([s], 0, steps=3)[0], b)
