"""The U-Net's plane-sweep convolutions and weight gradients at the edges of their tiles: planes smaller than a
tile, a ragged second tile, a depth past the accumulator ring and one plane at the bottom level, odd batches.

With arbitrary weights the BF16 roundings that FP32 against FP64 accumulation flips travel through the network, so
the comparison with the oracle has a wide tolerance that depends on the input.  Here every convolution row holds
one weight of 1 (a shifted copy of a channel) and the input is 0 or 1: activations are dyadic numbers of a few
bits, every product and sum is exact in FP32, and both sides round the same values.  What is left: the prediction
in FP32 (2^-24 relative per addition of the head: 1e-6), and for the gradients the FP32 value of the loss
derivative and of the slope 0.01, whose 2^-24 flips hardly any BF16 rounding; one flipped term of a sum changes it
by at most 2^-8 of that term (2^-8 of the layer's norm is allowed)."""
import numpy as np
import pytest

from oracle import learned_oracle as LO
from oracle import unet_oracle as UO

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rel(a, b):
    a, b = np.asarray(a, np.float64).ravel(), np.asarray(b, np.float64).ravel()
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def selecting_params(rng):
    p = []
    for w, b in UO.init_params(seed=5):
        s = np.zeros_like(w)
        if w.ndim == 5:
            for o in range(w.shape[0]):
                s[(o, rng.integers(w.shape[1])) + tuple(rng.integers(3, size=3))] = 1.0
        else:
            s[...] = rng.choice([-0.5, -0.25, 0.25, 0.5], size=w.shape)
        p.append((s, np.zeros_like(b)))
    return p


@pytest.mark.parametrize("shape", [(1, 8, 8, 8), (3, 8, 24, 8), (1, 8, 8, 136), (1, 40, 16, 8), (2, 16, 8, 40)])
def test_unet_at_tile_edges(shape):
    from paper_1703_01216_gb300 import fr3d as F
    B, D, Hh, W = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.integers(0, 2, size=(B, 1, D, Hh, W)).astype(np.float64)
    t = x + rng.integers(-4, 5, size=x.shape) * 0.125
    p = selecting_params(rng)
    y_ref, cache = UO.forward(p, x, rnd=LO.bf16_round)
    loss_ref, dy = UO.loss_and_grad(y_ref, t)
    g_ref = UO.backward(p, cache, dy, rnd=LO.bf16_round)
    net = F.Unet(D, Hh, W, B + 1, in_scale=1.0, seed=1)    # (room for a larger batch than is run)
    net.set_params(UO.pack(p).astype(np.float32))
    xd = torch.tensor(x[:, 0], dtype=torch.float32, device="cuda")
    td = torch.tensor(t[:, 0], dtype=torch.float32, device="cuda")
    y, grad, loss = torch.empty_like(xd), torch.empty(net.n_params, device="cuda"), torch.zeros(1, device="cuda")
    net.forward(xd, y)
    net.gradient(xd, td, grad, loss)
    torch.cuda.synchronize()
    assert net.error_flags() == 0
    assert rel(y.cpu(), y_ref[:, 0]) <= 1e-6
    assert abs(float(loss) - loss_ref) <= 1e-5 * loss_ref
    for (gw, gb), (rw, rb) in zip(UO.unpack(grad.double().cpu().numpy()), g_ref):
        assert rel(gw, rw) <= 2.0 ** -8 and rel(gb, rb) <= 2.0 ** -8
