"""Densities and total momentum straight from the bins (MIXED32), with particles in every place
they can be: stayers, outboxes, the overflow list (bins far too small), in few tiles shared
by several blocks and in many, alone and as a member of a batch. Against sums over the
particles that pic_particles returns, in the same precision (FP64 of the FP32 state).

Bound: a node's density is a sum of at most a few hundred positive terms, each rounded a few
times: 1e-13 of the largest; the momentum a sum of n terms against numpy's: 1e-12."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from runners import workload

pytestmark = pytest.mark.gpu


def _weights(order, d):
    d = np.abs(d)
    if order == 1:
        return np.maximum(0.0, 1.0 - d)
    if order == 2:
        return np.where(d < 0.5, 0.75 - d * d, 0.5 * np.maximum(0.0, 1.5 - d) ** 2)
    return np.where(d < 1.0, (4 - 6 * d * d + 3 * d ** 3) / 6, np.maximum(0.0, 2 - d) ** 3 / 6)


def _density(P, nx, ny, order, walls):
    out = np.zeros(nx * ny)
    bx, by = np.floor(P[0] - 0.5 * (order - 1)).astype(int), np.floor(P[1] - 0.5 * (order - 1)).astype(int)
    for b in range(order + 1):
        wy, row = _weights(order, P[1] - by - b), (by + b) % ny
        for a in range(order + 1):
            col, w = bx + a, wy * _weights(order, P[0] - bx - a)
            if walls:  # folded evenly; the unstored node x = nx is dropped
                col = np.where(col < 0, -col, np.where(col > nx, 2 * nx - col, col))
                w = np.where(col == nx, 0.0, w)
            np.add.at(out, row * nx + col % nx, w)
    return out.reshape(ny, nx)


@pytest.mark.parametrize("nx,ny,ppc,order,walls,tile,batch", [
    (64, 32, 20, 1, False, (32, 16), False), (72, 40, 5, 2, False, (8, 8), True), (50, 24, 8, 3, True, (16, 8), False),
    (256, 128, 4, 2, True, (8, 8), False)])
def test_density_and_momentum_from_every_storage(nx, ny, ppc, order, walls, tile, batch):
    w, sp, F0 = workload(nx, ny, ppc, gamma0=3.0, u_th=0.5, seed=91, field_amp=0.02, colocated=False)
    if walls:
        F0 = F0.copy()
        F0[1:4, :, 0] = 0.0
    mk = lambda **k: pic.pic_params_default(gamma0=3.0, precision=pic.PIC_MIXED32, **k)  # noqa: E731
    p = mk(nx=nx, ny=ny, ppc=ppc, shape_order=order, tile_x=tile[0], tile_y=tile[1], bin_slack=0.2,
           bc_x=pic.PIC_BC_WALLS if walls else pic.PIC_BC_PERIODIC)
    h = pic.pic_init_batch([mk(nx=24, ny=24, ppc=2), p] if batch else [p])
    try:
        pic.pic_select(h, 1 if batch else 0)
        for c in range(6):
            pic.pic_set_fields(h, c, np.ascontiguousarray(F0[c]).ravel())
        for s, d in enumerate(sp):
            pic.pic_load_particles(h, s, d["x"], d["y"], d["ux"], d["uy"], d["uz"])
        pic.pic_step(h, 3)
        P = [pic.pic_particles(h, s) for s in range(2)]
        cons = pic.pic_conservation(h)
        rho = [pic.fields_numpy(h, which, nx, ny) for which in (pic.PIC_DENSITY_P, pic.PIC_DENSITY_E)]
        both = pic.fields_numpy(h, pic.PIC_RHO, nx, ny)
        mw = pic.pic_moments(h)["macro_weight"]
    finally:
        pic.pic_free(h)
    ref = [_density(x, nx, ny, order, walls) for x in P]
    for a, b in zip(rho, ref):
        assert np.abs(a - b).max() <= 2e-6 * b.max()  # (positions come back as cell + FP32 offset, in FP64)
        assert abs(a.sum() - b.sum()) <= 1e-9 * b.sum()
    assert np.abs(both - mw * (rho[0] - rho[1])).max() <= 1e-13 * mw * rho[0].max()
    mom = mw * sum(x[2:].sum(axis=1) for x in P)
    np.testing.assert_allclose(cons["momentum"], mom, rtol=0, atol=1e-12 * mw * np.abs(P[0][2:]).sum())
