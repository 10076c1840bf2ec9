"""The U-Net's plane-sweep convolutions and weight gradients at the edges of their tiles: planes smaller than a
tile, a ragged second tile, a depth past the accumulator ring and one plane at the bottom level, odd batches
(tolerances as derived in test_gpu_unet.py: the same BF16 storage and FP32 accumulation)."""
import numpy as np
import pytest

from oracle import unet_oracle as UO

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rel(a, b):
    a, b = np.asarray(a, np.float64).ravel(), np.asarray(b, np.float64).ravel()
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("shape", [(1, 8, 8, 8), (3, 8, 24, 8), (1, 8, 8, 136), (1, 40, 16, 8), (2, 16, 8, 40)])
def test_unet_matches_the_oracle_at_tile_edges(shape):
    from paper_1703_01216_gb300 import fr3d as F
    B, D, Hh, W = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((B, 1, D, Hh, W)) * 0.5
    t = x + 0.2 * rng.standard_normal(x.shape)
    p = UO.init_params(seed=5)
    p[-1] = (rng.standard_normal((1, 16)) * 0.3, rng.standard_normal(1) * 0.05)
    p = [(w, b + 0.02 * rng.standard_normal(b.shape)) for w, b in p]
    flat = UO.pack(p).astype(np.float32)
    p32 = UO.unpack(flat.astype(np.float64))
    y_ref, cache = UO.forward(p32, x, rnd=UO_round)
    loss_ref, dy = UO.loss_and_grad(y_ref, t)
    g_ref = UO.backward(p32, cache, dy, rnd=UO_round)
    net = F.Unet(D, Hh, W, B + 1, in_scale=1.0, seed=1)    # (room for a larger batch than is run)
    net.set_params(flat)
    xd = torch.tensor(x[:, 0], dtype=torch.float32, device="cuda")
    td = torch.tensor(t[:, 0], dtype=torch.float32, device="cuda")
    y, grad, loss = torch.empty_like(xd), torch.empty(net.n_params, device="cuda"), torch.zeros(1, device="cuda")
    net.forward(xd, y)
    net.gradient(xd, td, grad, loss)
    torch.cuda.synchronize()
    assert net.error_flags() == 0
    assert rel(y.cpu(), y_ref[:, 0]) <= 1e-3
    assert abs(float(loss) - loss_ref) <= 1e-4 * loss_ref
    for (gw, gb), (rw, rb) in zip(UO.unpack(grad.double().cpu().numpy()), g_ref):
        assert rel(gw, rw) <= 3e-2 and rel(gb, rb) <= 3e-2


def UO_round(v):
    from oracle import learned_oracle as LO
    return LO.bf16_round(v)
