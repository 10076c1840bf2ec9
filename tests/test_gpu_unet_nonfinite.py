"""Non-finite values in the U-Net: a sample whose target is zero (the loss divides by its norm) makes the loss
infinite and gradients with NaN, and never hides behind finite values in the first layers' bias alone; the stored
BF16 values of NaN and infinity are those of the library's integer rounding, in every kernel that stores them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_zero_target_gives_an_infinite_loss_and_nonfinite_gradients():
    from paper_1703_01216_gb300 import fr3d as F
    rng = np.random.default_rng(1)
    net = F.Unet(8, 24, 32, 2, 1.0, 1)
    net.set_params((rng.standard_normal(net.n_params) * 0.05).astype(np.float32))
    x = torch.tensor(rng.standard_normal((2, 8, 24, 32)), dtype=torch.float32, device="cuda")
    t = 0.5 * x
    t[0] = 0
    g, loss = torch.zeros(net.n_params, device="cuda"), torch.zeros(1, device="cuda")
    net.gradient(x, t, g, loss)
    torch.cuda.synchronize()
    assert torch.isinf(loss).all() and float(loss) > 0
    bad = ~torch.isfinite(g)
    assert bool(bad.any()) and bool(bad[-17:].all())    # the head sees the infinite derivative directly
    # an untouched batch afterwards is finite again (nothing non-finite is left in the network's buffers)
    net.gradient(x, 0.5 * x, g, loss)
    torch.cuda.synchronize()
    assert torch.isfinite(g).all() and torch.isfinite(loss).all()
