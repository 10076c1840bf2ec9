"""Weight gradients whose partial sums are spread over 1, 4 and 16 threads per element (below 32, below 128 and from
128 units of 64-voxel spans on), with spans that end inside a K step, both row counts of the MMA (16 and 32 output
channels) and both sides of the input ring's wrap.  The selecting weights make every activation exact; the bounds are
those of test_gpu_unet_tiles."""
import numpy as np
import pytest

from oracle import learned_oracle as LO
from oracle import unet_oracle as UO
from test_gpu_unet_tiles import rel, selecting_params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 8, 16, 8), (2, 16, 24, 24), (3, 24, 40, 56)])
def test_weight_gradient_units(shape):
    from paper_1703_01216_gb300 import fr3d as F
    B, D, Hh, W = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.integers(0, 2, size=(B, 1, D, Hh, W)).astype(np.float64)
    t = x + rng.integers(-4, 5, size=x.shape) * 0.125
    p = selecting_params(rng)
    y_ref, cache = UO.forward(p, x, rnd=LO.bf16_round)
    _, dy = UO.loss_and_grad(y_ref, t)
    g_ref = UO.backward(p, cache, dy, rnd=LO.bf16_round)
    net = F.Unet(D, Hh, W, B, in_scale=1.0, seed=1)
    net.set_params(UO.pack(p).astype(np.float32))
    xd = torch.tensor(x[:, 0], dtype=torch.float32, device="cuda")
    td = torch.tensor(t[:, 0], dtype=torch.float32, device="cuda")
    grad, loss = torch.empty(net.n_params, device="cuda"), torch.zeros(1, device="cuda")
    net.gradient(xd, td, grad, loss)
    torch.cuda.synchronize()
    assert net.error_flags() == 0
    for (gw, gb), (rw, rb) in zip(UO.unpack(grad.double().cpu().numpy()), g_ref):
        assert rel(gw, rw) <= 2.0 ** -8 and rel(gb, rb) <= 2.0 ** -8
