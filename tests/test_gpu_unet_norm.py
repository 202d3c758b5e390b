"""The network's input normalisation, s = rms of each sample, on both sides of the size up to which
one launch takes it (8,192 pixels) and at the smallest images: the output scales with the input
(exactly, by powers of two), each sample by its own s, an all-zero sample gives the network at
zero (s = 1), and the output is that of a network without normalisation on x / s."""
import numpy as np
import pytest

from oracle import unet as ounet
from paper_1511_08225_gb300 import binding_unet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tensor_cores", [True, False])
@pytest.mark.parametrize("h,w", [(1, 1), (1, 31), (3, 11), (32, 33), (64, 128), (90, 91), (91, 91), (128, 128)])
def test_samples_are_scaled_by_their_rms(h, w, tensor_cores):
    nb, rng = 4, np.random.default_rng(h * w)
    params = [(np.float32(a), np.float32(rng.normal(0, 0.1, b.shape))) for a, b in ounet.init_params(1, 8, seed=2)]
    nets = [binding_unet.UNet(1, 8, h, w, max_batch=nb, normalise=n, tensor_cores=tensor_cores) for n in (True, False)]
    for net in nets:
        net.set_params(params)
    x = rng.normal(1.0, 1.0, (nb, h, w)).astype(np.float32)
    x[1] = 2.0 ** 20 * x[0]
    x[2] = 0.0
    s = np.sqrt((x.astype(np.float64) ** 2).mean((1, 2))).astype(np.float32)
    s[2] = 1.0
    inv = np.float32(1.0) / s
    y, z = (torch.zeros((nb, h, w), device="cuda") for _ in range(2))
    nets[0].forward(torch.tensor(x, device="cuda"), y)
    nets[1].forward(torch.tensor(x * inv[:, None, None], device="cuda"), z)
    y, z = y.cpu().numpy(), z.cpu().numpy()
    assert np.array_equal(y[1], 2.0 ** 20 * y[0])
    assert np.array_equal(y[2], z[2])
    for k in (0, 3):  # (s may differ from numpy's by an ulp, and a value that it moves over a
        # rounding boundary of BF16 by 2^-9)
        assert np.abs(y[k] - z[k] * s[k]).max() <= (1e-2 if tensor_cores else 1e-5) * np.abs(y[k]).max()
    for net in nets:
        net.close()
