"""The tile kernels' work items (MIXED32): a tile pushed whole by one CTA and the same tile
pushed in parts by several give the same currents, fields and particles, bit for bit. How a
tile is split follows from what else fills the launch: alone, a small simulation is cut into
parts; beside a large simulation of the same shape order its tiles stay whole."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from runners import workload

pytestmark = pytest.mark.gpu


def _state(h, nx, ny):
    F = np.stack([pic.fields_numpy(h, c, nx, ny) for c in range(9)])
    P = []
    for s in range(2):
        p = pic.pic_particles(h, s)
        P.append(p[:, np.lexsort(p[::-1])])
    return F, P


def _load(h, sp, F0):
    for c in range(6):
        pic.pic_set_fields(h, c, np.ascontiguousarray(F0[c]).ravel())
    for s, d in enumerate(sp):
        pic.pic_load_particles(h, s, d["x"], d["y"], d["ux"], d["uy"], d["uz"])


# ragged tiles, windows wider than the grid, fewer particles than one part, walls
@pytest.mark.parametrize("nx,ny,ppc,order,walls", [(64, 64, 40, 1, False), (72, 40, 33, 2, False), (100, 24, 20, 3, True),
                                                   (8, 8, 70, 2, False), (48, 32, 1, 3, False)])
def test_split_and_whole_tiles_agree_bit_for_bit(nx, ny, ppc, order, walls):
    w, sp, F0 = workload(nx, ny, ppc, gamma0=3.0, u_th=0.3, seed=61, field_amp=0.05, colocated=False)
    if walls:
        F0 = F0.copy()
        F0[1:4, :, 0] = 0.0
    bc = pic.PIC_BC_WALLS if walls else pic.PIC_BC_PERIODIC
    mk = lambda **k: pic.pic_params_default(gamma0=3.0, shape_order=order, precision=pic.PIC_MIXED32, **k)  # noqa: E731
    small = mk(nx=nx, ny=ny, ppc=ppc, bc_x=bc)
    large = mk(nx=1024, ny=512, ppc=ppc + 8)  # more tiles than the device holds CTAs
    got = []
    for params in ([small], [small, large]):
        h = pic.pic_init_batch(params)
        try:
            _load(h, sp, F0)
            pic.pic_step(h, 3)
            got.append(_state(h, nx, ny))
        finally:
            pic.pic_free(h)
    np.testing.assert_array_equal(got[0][0], got[1][0])
    for a, b in zip(got[0][1], got[1][1]):
        np.testing.assert_array_equal(a, b)
