"""The U-Net's blocked tensor-core path (BF16 operands in blocks of 8 channels with a zero
frame) at the sizes where its tiles, runs and slices end, against the FP64 oracle with the
same BF16 rounding: rows longer and shorter than the 128-pixel tile, an odd number of
rows (a lone last row of the row pairs), a channel count whose last 16-channel slice is
half padding (24), output channels beyond one accumulator slice and input channels beyond
the resident rows (base 128: 768 -> 256 and 128 -> 512).

The bars are those of the tensor-core tests in test_gpu_unet.py, and for their reason: a
conv input that straddles a BF16 rounding boundary between FP32 and FP64 accumulation
rounds differently on the two sides."""
import numpy as np
import pytest

from oracle import unet as ounet
from paper_1511_08225_gb300 import binding_unet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 8, 3, 129, 2), (1, 16, 1, 1, 1), (2, 8, 6, 258, 1), (2, 24, 10, 34, 2), (3, 8, 4, 128, 1),
          (3, 128, 8, 12, 1)]


def _case(levels, base, h, w, nb):
    rng = np.random.default_rng(levels * 1000 + base + h * w)
    params = [(np.float32(a), np.float32(rng.normal(0, 0.1, b.shape)))
              for a, b in ounet.init_params(levels, base, seed=levels + base)]
    x, t = (rng.normal(size=(nb, h, w)).astype(np.float32) for _ in range(2))
    net = binding_unet.UNet(levels, base, h, w, max_batch=nb, normalise=False, tensor_cores=True)
    net.set_params(params)
    return [(ounet.bf16(a), b.astype(np.float64)) for a, b in params], x, t, net


@pytest.mark.parametrize("levels,base,h,w,nb", SHAPES)
def test_forward_and_gradients_at_the_edges_of_tiles(levels, base, h, w, nb):
    params, x, t, net = _case(levels, base, h, w, nb)
    y = torch.zeros((nb, h, w), device="cuda")
    net.forward(torch.tensor(x, device="cuda"), y)
    loss, grads = net.gradients(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"))
    got = y.cpu().numpy()
    ref, ref_loss = None, 0.0
    for k in range(nb):
        yk, cache = ounet.forward(params, x[k].astype(np.float64), levels, act_bf16=True)
        assert np.abs(got[k] - yk).max() <= 1e-2 * np.abs(yk).max(), k
        r = yk - t[k]
        ref_loss += float((r * r).sum()) / x.size
        g = ounet.backward(params, cache, 2.0 * r / x.size, levels, act_bf16=True)
        ref = g if ref is None else [(a + c, b + d) for (a, b), (c, d) in zip(ref, g)]
    assert loss == pytest.approx(ref_loss, rel=1e-3)
    for k, ((dw, db), (rw, rb)) in enumerate(zip(grads, ref)):
        assert np.abs(dw - rw).max() <= 1e-2 * np.abs(rw).max(), ("W", k)
        assert np.abs(db - rb).max() <= 1e-2 * max(np.abs(rb).max(), 1e-12), ("b", k)
    net.close()


def test_repeated_calls_leave_the_frames_zero():
    """Every layer writes only the pixels inside its frame, so a smaller batch, a repeat
    and a training step in between give the first call's output bit for bit."""
    params, x, t, net = _case(3, 16, 12, 20, 3)
    xd, td = torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda")
    first, again, one = (torch.zeros_like(xd) for _ in range(3))
    net.forward(xd, first)
    g0 = net.gradients(xd, td)
    net.forward(xd[:1].contiguous(), one[:1])
    net.forward(xd, again)
    g1 = net.gradients(xd, td)
    assert torch.equal(first, again) and torch.equal(first[:1], one[:1])
    assert g0[0] == g1[0]
    assert all(np.array_equal(a, c) and np.array_equal(b, d) for (a, b), (c, d) in zip(g0[1], g1[1]))
    net.close()
