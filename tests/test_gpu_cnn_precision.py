"""The network's gradients against 64-bit sums of the same BF16 operands, over batches whose
sums are a few and many accumulations long. The network passes its input through (one unit
weight per output channel), so every activation is the input's BF16 value and every output
gradient the loss's, rounded once; inputs and output gradients are positive, so a sum that is
cut short at every addition shows in full.

Bound, relative to the sum of magnitudes (here the sum itself): at most 48 additions in tensor
memory, the partial sum growing evenly, each off by less than 2^-23 of it: 24.5 * 2^-23; then
FP32 additions rounded to nearest: as many as a CTA has flushes (chunks of 64 pixels over 76
CTAs, 12 to a flush), 19 in each of four chains over the CTAs and 2 to join them, each off by
2^-24 at most. The bias: 12 additions per thread and flush, 5 lanes and 3 warps in place of the
tensor memory's."""
import numpy as np
import pytest

import paper_1412_2480_gb300 as pic

pytestmark = pytest.mark.gpu
LAYERS = [(3, 32), (32, 32), (32, 32), (32, 3)]


@pytest.mark.parametrize("nimg,nx,ny", [(1, 32, 32), (8, 64, 64), (5, 96, 128), (16, 128, 128), (16, 256, 256)])
def test_gradients_against_64_bit_sums(nimg, nx, ny):
    import torch
    params, offs, o = [], [], 0
    for L, (ci, co) in enumerate(LAYERS):
        W = np.zeros((co, 9, ci), dtype=np.float32)
        W[np.arange(co), 4, np.arange(co) % (3 if L == 0 else ci)] = 1.0
        params += [W.ravel(), np.zeros(co, dtype=np.float32)]
        offs.append((o, o + W.size, ci, co))
        o += W.size + co
    g = torch.Generator(device="cuda")
    g.manual_seed(nimg * 1000 + nx)
    x = 1.0 + torch.rand(nimg, 3, ny, nx, generator=g, device="cuda")
    t = torch.zeros_like(x)
    c = pic.pic_cnn_create()
    try:
        pic.pic_cnn_set_params(c, np.concatenate(params))
        grad, _ = pic.pic_cnn_gradient(c, x.cpu().numpy(), t.cpu().numpy())
    finally:
        pic.pic_cnn_free(c)
    npix = nimg * nx * ny
    X = x.bfloat16()
    scale = float(np.float32(2.0) / np.float32(3 * npix))
    dY = (X.float() * scale).bfloat16().double()
    X = X.double()
    W = torch.stack([torch.einsum("nkyx,ncyx->kc", dY, torch.roll(X, (1 - tap // 3, 1 - tap % 3), (2, 3)))
                     for tap in range(9)], 1).cpu().numpy()  # [output channel][tap][input channel]
    b = dY.sum((0, 2, 3)).cpu().numpy()
    flushes = -(-(npix // 64) // (76 * 12))
    joins = (flushes + 19 + 2) * 2.0 ** -24
    for w0, b0, ci, co in offs:
        got = grad[w0:b0].reshape(co, 9, ci).astype(np.float64)
        want = np.zeros((co, 9, ci))
        want[:3] = W[:, :, np.arange(ci) % 3]
        assert np.all(got[3:] == 0.0)
        assert np.abs(got[:3] / want[:3] - 1.0).max() <= 24.5 * 2.0 ** -23 + joins
        gb = grad[b0:b0 + co].astype(np.float64)
        assert np.all(gb[3:] == 0.0)
        assert np.abs(gb[:3] / b - 1.0).max() <= (12 + 5 + 3) * 2.0 ** -24 + joins


def test_gradient_after_a_wait_that_ran_out_is_the_same_to_the_bit():
    rng = np.random.default_rng(5)
    x, t = (rng.standard_normal((2, 3, 64, 64)).astype(np.float32) for _ in range(2))
    c = pic.pic_cnn_create()
    try:
        pic.pic_cnn_set_params(c, (rng.standard_normal(pic.PIC_CNN_NPARAMS) * 0.05).astype(np.float32))
        want, loss = pic.pic_cnn_gradient(c, x, t)
        pic.pic_cnn_set_wait_limit(c, 1)
        with pytest.raises(pic.PicError) as e:
            pic.pic_cnn_gradient(c, -2 * x, t)
        assert e.value.code == pic.PIC_ETIMEOUT, e.value
        pic.pic_cnn_set_wait_limit(c, 0)
        got, loss2 = pic.pic_cnn_gradient(c, x, t)
        np.testing.assert_array_equal(got, want)
        assert loss2 == pytest.approx(loss, rel=1e-12)
    finally:
        pic.pic_cnn_free(c)
