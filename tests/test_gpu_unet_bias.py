"""The bias gradients of the tensor-core convolutions are FP64 sums of the unrounded output
gradient, or as good.  A network of one level whose output convolution passes its input on (one
tap), so that the first convolution's output gradient is the loss's: single pixels of chosen
size, exact in BF16.  Sums that fit in 53 bits come
out exactly whatever lies between them, and an infinite or huge gradient gives what FP64 gives."""
import numpy as np
import pytest

from paper_1511_08225_gb300 import binding_unet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H, W, BASE = 4, 32, 8


def _bias_gradient(pixels, weight=1.0, taps=np.s_[1, 1]):
    """pixels: {(y, x): output gradient}; the bias gradient of the first convolution, whose
    output gradient is the loss's through these taps of this weight."""
    w_in = np.zeros((BASE, 1, 3, 3), np.float32)
    w_out = np.zeros((1, BASE, 3, 3), np.float32)
    w_out[(slice(None), slice(None), *taps)] = weight
    net = binding_unet.UNet(1, BASE, H, W, max_batch=1, normalise=False, tensor_cores=True)
    net.set_params([(w_in, np.ones(BASE, np.float32)), (w_out, np.full(1, -BASE * weight, np.float32))])
    x = torch.zeros((1, H, W), device="cuda")
    t = torch.zeros_like(x)
    net.forward(x, t)  # the target is the output but at those pixels
    for (i, j), g in pixels.items():
        t[0, i, j] -= g * (H * W / 2)
    _, grads = net.gradients(x, t)
    net.close()
    return np.array(grads[0][1])


@pytest.mark.parametrize("small", [1.0, 2.0 ** -2])
@pytest.mark.parametrize("lanes", [(0, 16, 8, 4, 20), (0, 1, 2, 3, 4), (31, 15, 7, 3, 30)])
def test_terms_of_three_sizes_cancel_exactly(small, lanes):
    big, mid = 2.0 ** 50, 2.0 ** 25
    b, m, s, nb, nm = lanes
    got = _bias_gradient({(0, b): big, (0, m): mid, (0, s): small, (0, nb): -big, (0, nm): -mid})
    assert (got == small).all()
    got = _bias_gradient({(0, b): big, (1, m): mid, (1, s): small, (1, nb): -big, (0, nm): -mid})
    assert (got == small).all()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_a_gradient_that_is_not_finite(value):
    got = _bias_gradient({(1, 5): value, (2, 9): 1.0}, taps=np.s_[:, :])
    assert np.array_equal(got, np.full(BASE, value, np.float32), equal_nan=True)


def test_partial_sums_beyond_fp32s_range():
    g = 2.0 ** 116  # times the weight 2^124: sixteen of them pass FP32's largest number
    pixels = {(i, j): g if i < 2 else -g for i in range(H) for j in range(W)}
    del pixels[3, 17]
    assert (_bias_gradient(pixels, weight=256.0) == g * 256.0).all()
