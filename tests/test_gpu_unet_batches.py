"""Gradients of a batch in networks made for larger batches: the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def data(shape, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.rand(shape, generator=gen, device="cuda")
    return x, x + 0.1 * torch.rand(shape, generator=gen, device="cuda")


def network(F, shape, max_batch):
    net = F.Unet(*shape, max_batch, in_scale=4.0, seed=3)
    p = net.get_params()
    p[-17:] = 0.1 * np.random.default_rng(1).standard_normal(17)   # (a new network's head is zero)
    net.set_params(p)
    return net


def gradient(net, x, t):
    g, l = torch.zeros(net.n_params, device="cuda"), torch.zeros(1, device="cuda")
    net.gradient(x, t, g, l)
    torch.cuda.synchronize()
    assert net.error_flags() == 0
    return g, l


@pytest.mark.parametrize("shape,B,more", [((8, 64, 64), 2, (3, 9, 16)), ((16, 24, 40), 1, (16,)), ((8, 96, 96), 3, (4,))])
def test_gradient_bits_do_not_depend_on_the_largest_batch(shape, B, more):
    from paper_1703_01216_gb300 import fr3d as F
    x, t = data((B, *shape), sum(shape))
    ref = gradient(network(F, shape, B), x, t)
    for m in more:
        net = network(F, shape, m)
        xm, tm = data((m, *shape), 5)
        for _ in range(2):   # before and after a batch of another size
            got = gradient(net, x, t)
            assert all(torch.equal(a, b) for a, b in zip(got, ref))
            gradient(net, xm, tm)
