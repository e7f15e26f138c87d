"""The FP64 PCG's cooperative kernel in each of its forms (one cell per thread, two cells per
thread, vectors in memory), at the sizes where a form begins or ends on 152 SMs: one step
against the oracle's plain CG, periodic and walled.

Bound: both sides stop at ||r|| <= 1e-13 ||b||, so their solutions differ by at most
2e-13 kappa(A) <= 1e-12 in norm at CFL 0.7, theta 1/2 (kappa = 1 + 8 (theta cfl)^2 < 2)."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from runners import check, run_gpu, run_oracle, workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,walls", [(8, 8, False), (17, 15, True), (342, 341, False), (343, 341, True),
                                         (400, 389, False), (401, 389, True), (512, 320, False)])
def test_cg_forms_match_the_oracle(nx, ny, walls):
    w, sp, F0 = workload(nx, ny, 1, gamma0=3.0, u_th=0.1, seed=71, field_amp=0.05, colocated=False)
    if walls:
        F0 = F0.copy()
        F0[1:4, :, 0] = 0.0
    bc = pic.PIC_BC_WALLS if walls else pic.PIC_BC_PERIODIC
    F, _, m = run_gpu(nx, ny, 1, sp, F0, 1, 1, cfl=0.7, gamma0=3.0, cg_rtol=1e-13, bc_x=bc, want_particles=False)
    ref, _, _ = run_oracle(nx, ny, w, sp, F0, 1, 1, cfl=0.7, cg_rtol=1e-13, walls=walls)
    assert 0 < m["cg_rel_resid"] <= 1e-13
    for c in range(12):
        if np.linalg.norm(ref[c]) > 0:
            check(F[c], ref[c], 1e-12 if c < 9 else 2e-12, f"component {c}")
