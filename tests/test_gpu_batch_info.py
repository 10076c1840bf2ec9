"""Info words of a batched plan: a bounded wait of the tile queue that gives up (its column tiles withhold the counts
that release the intermediate, so the row tiles' waits run out after about a second) is reported to every instance of
the launch that has a word, whatever its alpha rule; the next run overwrites the words and is exact."""
import time

import pytest

from paper_1703_01216_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def F():
    from paper_1703_01216_gb300 import fr3d
    prev = fr3d.autotune_mode()
    yield fr3d
    fr3d.autotune_mode(prev)
    fr3d.test_withhold_queue_counts(False)


def test_every_instance_reports_a_wait_that_gave_up(F):
    shapes = [(96, 3, 1, "rule"), (96, 5, 2, "fixed"), (256, 2, 1, "given"), (256, 3, 2, "none"), (96, 2, 2, "rule")]
    items, words, refs = [], [], []
    for k, (n, mp, q, kind) in enumerate(shapes):
        w = I.make_workload(n, mp, q=q, n_incl=1, n_alpha=12, seed=800 + k)
        H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
        U = torch.as_tensor(w.noise, dtype=torch.float32, device="cuda")
        info = None if kind == "none" else torch.full((1,), 0x40, dtype=torch.int32, device="cuda")
        if kind == "fixed":
            opts = F.Opts(alpha=1e-3, points=w.sources, info=info)
        elif kind == "given":
            opts = F.Opts(alphas=w.alphas, given=True, points=w.sources, info=info,
                          alpha_idx=torch.full((1,), 3, dtype=torch.int32, device="cuda"))
        else:
            opts = F.Opts(alphas=w.alphas, delta=0.3 * float(U.norm()), points=w.sources, info=info)
        items.append((H, U, q, opts, torch.empty((mp, n, n), device="cuda")))
        words.append(info)
    plan = F.Batch(items)
    F.autotune_mode(2 + 3)
    plan.run()
    torch.cuda.synchronize()
    refs = [it[4].clone() for it in items]
    assert all(i is None or not int(i) & (0x40 | F.INFO_TIMEOUT) for i in words)
    F.autotune_mode(2 + 5)
    F.test_withhold_queue_counts(True)
    t0 = time.perf_counter()
    plan.run()
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 < 30.0
    F.test_withhold_queue_counts(False)
    assert all(i is None or int(i) & F.INFO_TIMEOUT for i in words)
    plan.run()
    torch.cuda.synchronize()
    for it, ref, i in zip(items, refs, words):
        assert torch.equal(it[4], ref)
        assert i is None or not int(i) & F.INFO_TIMEOUT
