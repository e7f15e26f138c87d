"""Whole against split tiles (MIXED32): beside a simulation of 4096 equally full tiles the tiles
of a small one stay whole, alone each is cut into parts (tests/test_tile_plan.py evaluates the
rule for these sizes). Fields, currents and particles are the same, bit for bit: with the slot
counters of the next buffer in shared memory or in global memory, and with one current window
or several. And a tile fuller than its bins were sized for, whose parts take equal shares."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from runners import workload

pytestmark = pytest.mark.gpu


def _run(params, sp, F0, nx, ny, steps=3):
    h = pic.pic_init_batch(params)
    try:
        for c in range(6):
            pic.pic_set_fields(h, c, np.ascontiguousarray(F0[c]).ravel())
        for s, d in enumerate(sp):
            pic.pic_load_particles(h, s, d["x"], d["y"], d["ux"], d["uy"], d["uz"])
        pic.pic_step(h, steps)
        F = np.stack([pic.fields_numpy(h, c, nx, ny) for c in range(9)])
        P = [pic.pic_particles(h, s) for s in range(2)]
        return F, [p[:, np.lexsort(p[::-1])] for p in P]
    finally:
        pic.pic_free(h)


def _same(a, b):
    np.testing.assert_array_equal(a[0], b[0])
    for x, y in zip(a[1], b[1]):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("nx,ny,order,walls", [(64, 64, 1, False), (72, 40, 2, False), (100, 24, 3, True), (72, 40, 1, True)])
def test_whole_and_split_tiles_agree_bit_for_bit(nx, ny, order, walls):
    w, sp, F0 = workload(nx, ny, 12, gamma0=3.0, u_th=0.3, seed=62, field_amp=0.05, colocated=False)
    if walls:
        F0 = F0.copy()
        F0[1:4, :, 0] = 0.0
    mk = lambda **k: pic.pic_params_default(gamma0=3.0, shape_order=order, ppc=12, precision=pic.PIC_MIXED32, **k)  # noqa: E731
    small = mk(nx=nx, ny=ny, bc_x=pic.PIC_BC_WALLS if walls else pic.PIC_BC_PERIODIC)
    _same(_run([small], sp, F0, nx, ny), _run([small, mk(nx=2048, ny=1024)], sp, F0, nx, ny))


@pytest.mark.parametrize("slack", [0.2, 4.0])
def test_bins_of_another_size_give_the_same_bits(slack):
    nx, ny = 72, 40
    w, sp, F0 = workload(nx, ny, 40, gamma0=3.0, u_th=0.3, seed=63, field_amp=0.05, colocated=False)
    mk = lambda **k: pic.pic_params_default(nx=nx, ny=ny, gamma0=3.0, shape_order=2, precision=pic.PIC_MIXED32, **k)  # noqa: E731
    _same(_run([mk(ppc=40)], sp, F0, nx, ny), _run([mk(ppc=40, bin_slack=slack)], sp, F0, nx, ny))
    # three times as many particles as the simulation was sized for, cut in two ways
    under = mk(ppc=13, bin_slack=8.0)
    other = pic.pic_params_default(nx=2048, ny=512, ppc=12, gamma0=3.0, shape_order=2, precision=pic.PIC_MIXED32)
    _same(_run([under], sp, F0, nx, ny), _run([under, other], sp, F0, nx, ny))
