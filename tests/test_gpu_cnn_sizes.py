"""The network's gradients over the sizes their kernels cut differently: fewer chunks of 64
pixels than CTAs per layer (down to two), one more than a multiple, two rounds and more per
CTA, and images whose rows are shorter than a chunk or no multiple of it. With one +-1 weight
per output channel, inputs in {-1, 0, 1} and targets that make the output gradient an integer,
every activation, gradient and sum is a small integer (exact in BF16 and FP32 in any order),
so the result equals the oracle's element by element; and a random network's gradient is the
same to the bit when it is computed twice."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic
from oracle import cnn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nimg,nx,ny", [(1, 8, 16), (3, 8, 16), (1, 48, 40), (5, 24, 16), (1, 64, 154), (2, 64, 160),
                                        (8, 96, 128)])
def test_gradients_over_sizes(nimg, nx, ny):
    rng = np.random.default_rng(nimg * 1000 + nx)
    p = np.zeros(cnn.NPARAMS)
    for (ci, co), (wo, bo) in zip(cnn.LAYERS, cnn.offsets()):
        for o in range(co):
            p[wo + o * 9 * ci + rng.integers(0, 9 * ci)] = rng.choice((-1.0, 1.0))
    b = rng.integers(-1, 2, (nimg, 3, ny, nx)).astype(np.float64)
    out = cnn.forward(p, b, quantize=True)
    t = out - rng.integers(-1, 2, out.shape) * 1.5 * nimg * nx * ny
    _, ref = cnn.loss_and_grad(p, b, t, quantize=True)
    assert np.abs(ref).max() > 0
    q = (rng.standard_normal(cnn.NPARAMS) * 0.06).astype(np.float32)
    c = pic.pic_cnn_create()
    try:
        pic.pic_cnn_set_params(c, p.astype(np.float32))
        g, _ = pic.pic_cnn_gradient(c, b.astype(np.float32), t.astype(np.float32))
        pic.pic_cnn_set_params(c, q)
        twice = [pic.pic_cnn_gradient(c, b.astype(np.float32), (0.5 * b).astype(np.float32))[0] for _ in range(2)]
    finally:
        pic.pic_cnn_free(c)
    np.testing.assert_array_equal(g, ref.astype(np.float32))
    np.testing.assert_array_equal(twice[0], twice[1])
