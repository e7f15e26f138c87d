"""The kinetic energy of FP64 particles: gamma is the correctly rounded square root of
1 + u^2. Momenta whose squares are exact and 64 equal pairs without fields make every other
step exact or a rounding that is known here (a doubling, a sum of equal terms, one subtraction,
one product with the particle weight), so the result is the host's to the bit."""
import math

import numpy as np
import pytest

import paper_1412_2480_gb300 as pic

pytestmark = pytest.mark.gpu


def test_kinetic_energy_to_the_last_place():
    n = 64
    h = pic.pic_init(pic.pic_params_default(nx=16, ny=16, ppc=1, gamma0=2.0, shape_order=1, precision=pic.PIC_FP64,
                                            flags=pic.PIC_NO_DEPOSIT))
    try:
        w = pic.pic_moments(h)["macro_weight"]
        rng = np.random.default_rng(3)
        x, y = rng.uniform(2, 14, n), rng.uniform(2, 14, n)
        z = np.zeros(n)
        for u in rng.integers(1, 5000, (150, 3)).astype(np.float64):
            for s in range(2):
                pic.pic_load_particles(h, s, x, y, z + u[0], z + u[1], z + u[2])
            pic.pic_step(h, 1)
            gamma = math.sqrt(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
            assert pic.pic_moments(h)["U_K"] == 2 * (0.5 * w * (n * (2.0 * gamma - 2.0))), (u, gamma)
    finally:
        pic.pic_free(h)
