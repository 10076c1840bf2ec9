"""The U-Net's programmatic launches: calls that follow each other without a wait, with other inputs each time, and
replays of a captured gradient give the bits of the same calls run one at a time."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 8, 8, 8), (2, 16, 24, 40), (3, 8, 64, 64)])
def test_unet_calls_back_to_back(shape):
    from paper_1703_01216_gb300 import fr3d as F
    B, D, Hh, W = shape
    gen = torch.Generator(device="cuda")
    gen.manual_seed(sum(shape))
    net = F.Unet(D, Hh, W, B, in_scale=4.0, seed=3)
    p = net.get_params()
    p[-17:] = 0.1 * np.random.default_rng(1).standard_normal(17)   # (a new network's head is zero)
    net.set_params(p)
    xs = [torch.rand((B, D, Hh, W), generator=gen, device="cuda") for _ in range(6)]
    ts = [x + 0.1 * torch.rand(x.shape, generator=gen, device="cuda") for x in xs]

    def outputs():
        return [(torch.zeros_like(x), torch.zeros(net.n_params, device="cuda"), torch.zeros(1, device="cuda")) for x in xs]

    want, got = outputs(), outputs()
    for x, t, (y, g, l) in zip(xs, ts, want):
        net.forward(x, y)
        torch.cuda.synchronize()
        net.gradient(x, t, g, l)
        torch.cuda.synchronize()
    for x, t, (y, g, l) in zip(xs, ts, got):
        net.forward(x, y)
        net.gradient(x, t, g, l)
    torch.cuda.synchronize()
    for a, b in zip(want, got):
        assert all(torch.equal(u, v) for u, v in zip(a, b))
    x, t = xs[0].clone(), ts[0].clone()
    y, g, l = outputs()[0]
    s = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        net.forward(x, y, stream=s)
        net.gradient(x, t, g, l, stream=s)
    for k in (3, 1, 4):
        x.copy_(xs[k])
        t.copy_(ts[k])
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(u, v) for u, v in zip((y, g, l), want[k]))
    assert net.error_flags() == 0
