"""Gradients of a batch in networks made for larger batches (the same bits), and against those of its samples: every way
of adding the units' partial sums (1, 4, 16 and 32 threads per element) and of walking a unit (one and several
sub-ranges of 128 positions)."""
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


@pytest.mark.parametrize("shape,threads", [((32, 64, 64), {1, 4, 16, 32}), ((8, 104, 104), {1, 4, 16})])
def test_batch_gradient_is_the_mean_of_its_samples(shape, threads):
    """A batch of 16: the loss is the mean over the samples, and 1 / 16 scales every stored value exactly, so the batch's
    gradient is the mean of the samples' up to the order of FP32 sums: at most 256 chained accumulations of 2^-23 of the
    running sum each, 2^-15 of the terms' magnitudes, times 16 for cancellation among them: 2^-11.  A sample alone has
    fewer than 128 units of one sub-range, which the oracle tests cover.  A lost unit of 528 would be 2^-9 if all units
    were alike, more if their signs differ."""
    from paper_1703_01216_gb300 import fr3d as F
    B = 16
    net = network(F, shape, B)
    plans = [net.test_wgrad_plan(k, B) for k in range(15)]
    assert {32 if u >= 512 else 16 if u >= 128 else 4 if u >= 32 else 1 for u, _ in plans} == threads
    assert max(s for _, s in plans) >= 384
    assert all(u < 128 and s == 128 for u, s in (net.test_wgrad_plan(k, 1) for k in range(15)))
    x, t = data((B, *shape), sum(shape))
    got = gradient(net, x, t)[0].double()
    ref = sum(gradient(net, x[b:b + 1].contiguous(), t[b:b + 1].contiguous())[0].double() for b in range(B)) / B
    at, layers = 0, [(16, 1), (16, 16), (32, 16), (32, 32), (64, 32), (64, 64), (128, 64), (128, 128), (128, 128),
                     (64, 192), (64, 64), (32, 96), (32, 32), (16, 48), (16, 16)]
    for co, ci in layers:
        for n in (co * ci * 27, co):
            a, b = got[at:at + n], ref[at:at + n]
            assert float((a - b).norm()) <= 2.0 ** -11 * float(b.norm()), (co, ci, n)
            at += n
    assert float((got[at:] - ref[at:]).norm()) <= 2.0 ** -11 * float(ref[at:].norm())
