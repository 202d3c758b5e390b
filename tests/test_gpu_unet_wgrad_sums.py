"""The tensor-core weight gradient adds its pixel ranges in FP64, a range's products in FP32: a
range must not be longer than the 256 pixels that the convolution with 128 -> 256 channels has
had at 64 x 64.  Products of integers below 2^16 then stay exact in the range's sum (below
2^24), and with signs that keep the whole sum small the gradient is the integer sum."""
import numpy as np
import pytest

from paper_1511_08225_gb300 import binding_unet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_products_of_a_range_stay_exact():
    nb, hw, base = 2, 128, 128
    rng = np.random.default_rng(4)
    shapes = binding_unet.layer_shapes(2, base)
    params = [(np.zeros((co, ci, 3, 3), np.float32), np.zeros(co, np.float32)) for ci, co in shapes]
    params[0][0][0, 0, 1, 1] = 1.0   # e_0[0] = x, constant over 2 x 2 pixels: its pool is x
    params[1][1][0] = 1.0            # e_1[0] = 1
    params[2][0][0, 0, 1, 1] = 1.0   # d_0[0] = up(e_1)[0]
    params[3][0][0, 0, 1, 1] = 1.0   # y = d_0[0] - 1 = 0
    params[3][1][0] = -1.0
    net = binding_unet.UNet(2, base, hw, hw, max_batch=nb, normalise=False, tensor_cores=True)
    net.set_params(params)
    a = rng.integers(192, 256, (nb, hw // 2, hw // 2))           # conv 1's input
    g = rng.integers(192, 256, (nb, hw // 2, hw // 2))           # its output gradient
    g[:, hw // 4:] *= -1
    x = a.repeat(2, 1).repeat(2, 2).astype(np.float32)
    t = np.zeros((nb, hw, hw), np.float32)
    t[:, ::2, ::2] = -g * (nb * hw * hw / 2)                     # the loss's gradient: g at one of four pixels
    loss, grads = net.gradients(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"))
    want = int((a * g).sum())
    assert abs(want) < 1 << 24
    assert grads[1][0][0, 0, 1, 1] == want
    assert grads[1][1][0] == int(g.sum())
    net.close()
