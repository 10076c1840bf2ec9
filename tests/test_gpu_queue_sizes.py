"""The tile queue at its radix-3 and smaller sizes: the same bits as the register tile (variant 3) for single calls
(depth counts below and above the queue's lag, source counts around its halves, bands) and for a batch of instances
of several sizes, whose tickets run across instances; repeated, since the ordering depends on timing."""
import pytest

from paper_1703_01216_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_1703_01216_gb300 import fr3d
    prev = fr3d.autotune_mode()
    yield fr3d
    fr3d.autotune_mode(prev)


@pytest.mark.parametrize("n,mp,q,nb", [(96, 1, 1, 1), (96, 33, 3, 4), (96, 200, 2, 1), (128, 5, 1, 1), (128, 64, 4, 8),
                                       (192, 1, 2, 1), (192, 51, 5, 8), (192, 9, 1, 1)])
def test_sizes_match_the_register_tile(F, n, mp, q, nb):
    w = I.make_workload(n, mp, q=q, n_incl=1, n_alpha=12, seed=n + mp)
    H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
    U = torch.as_tensor(w.noise, dtype=torch.float32, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    opts = F.Opts(alphas=w.alphas, delta=0.3 * float(U.norm()), points=w.sources, n_bands=nb, info=info)
    outs = {}
    for v, reps in ((3, 1), (5, 6)):
        F.autotune_mode(2 + v)
        for _ in range(reps):
            out = torch.full((mp, n, n), float("nan"), device="cuda")
            F.invert(H, U, q, out, opts)
            torch.cuda.synchronize()
            assert F.autotune_query(H)[0] == v and not int(info) & F.INFO_TIMEOUT
            outs.setdefault(v, out)
            assert torch.equal(out, outs[3])


def test_batched_queues_match_the_register_tile(F):
    shapes = [(96, 16, 2), (192, 3, 1), (128, 48, 3), (96, 1, 1), (192, 20, 4), (128, 7, 1), (256, 5, 2), (96, 40, 5),
              (256, 33, 1), (192, 2, 2)]
    items, refs = [], []
    for k, (n, mp, q) in enumerate(shapes):
        w = I.make_workload(n, mp, q=q, n_incl=1, n_alpha=12, seed=700 + k)
        H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
        U = torch.as_tensor(w.noise, dtype=torch.float32, device="cuda")
        opts = F.Opts(alphas=w.alphas, delta=0.3 * float(U.norm()), points=w.sources)
        out = torch.empty((mp, n, n), device="cuda")
        F.autotune_mode(2 + 3)
        F.invert(H, U, q, out, opts)
        torch.cuda.synchronize()
        refs.append(out.clone())
        items.append((H, U, q, opts, out))
    plan = F.Batch(items)
    for mode in (2 + 5, 2 + 5, 2 + 5, 1, 1):
        F.autotune_mode(mode)
        for it in items:
            it[4].fill_(float("nan"))
        plan.run()
        torch.cuda.synchronize()
        for it, ref in zip(items, refs):
            assert torch.equal(it[4], ref)
