"""Calls on a device without room (fr3d_test_alloc_budget makes requests fail as if it were full): what a handle or a plan
can do without is given up before a call fails, and results stay those of a call with room."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1703_01216_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture
def F():
    from paper_1703_01216_gb300 import fr3d
    prev = fr3d.autotune_mode()
    yield fr3d
    fr3d.test_alloc_budget(-1)
    fr3d.autotune_mode(prev)


def least(F, call, step, top):
    """The smallest budget (a multiple of step) with which call(budget) does not run out of memory."""
    for b in range(0, top, step):
        try:
            call(b)
            return b
        except F.Fr3dError:
            pass
        finally:
            F.test_alloc_budget(-1)
    raise AssertionError("no budget was enough")


@pytest.mark.parametrize("n,prec,mp", [(64, 1, 8), (512, 0, 3)])
def test_weights_make_room_for_the_workspace(F, n, prec, mp):
    dt = torch.float64 if prec == F.PREC_FP64 else torch.float32
    w = I.make_workload(n, mp, q=3, n_incl=1, seed=71)
    U = torch.as_tensor(w.noise, dtype=dt, device="cuda")
    pts = np.asarray(w.sources)
    ref = torch.empty((mp, n, n), dtype=dt, device="cuda")
    F.invert(F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu), U, 3, ref, F.Opts(alpha=1e-2, precision=prec, points=pts))
    outs = []

    def grow(first):
        def call(budget):
            H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
            if first == "xi":   # one source's weights are kept
                F.invert(H, U[:1].contiguous(), 1, torch.empty_like(ref), F.Opts(alpha=1e-2, precision=prec, points=pts[:1]))
            else:
                z = torch.empty((1, mp, n, n), dtype=dt, device="cuda")
                F.invert(H, U[:1].contiguous(), 1, z, F.Opts(alpha=1e-2, precision=prec, output=F.OUT_ZETA))
            torch.cuda.synchronize()
            F.test_alloc_budget(budget)
            out = torch.empty_like(ref)
            F.invert(H, U, 3, out, F.Opts(alpha=1e-2, precision=prec, points=pts))
            torch.cuda.synchronize()
            outs.append(out)
        return call

    table = U.element_size() * mp * n * n
    step = table // 8
    kept, none = (least(F, grow(first), step, 64 * table) for first in ("xi", "zeta"))
    assert kept <= none - table + step, (kept, none, table)
    for out in outs:   # (the weights may be evaluated per voxel: a few ulp)
        assert float((out - ref).norm()) <= 32 * torch.finfo(dt).eps * float(ref.norm())


def test_weights_without_room_are_asked_for_once_per_source_set(F):
    n, mp = 48, 4
    w = I.make_workload(n, mp, q=2, n_incl=1, seed=72)
    pts = np.asarray(w.sources)
    U = torch.as_tensor(w.noise, dtype=torch.float64, device="cuda")
    out, z = torch.empty((mp, n, n), dtype=U.dtype, device="cuda"), torch.empty((2, mp, n, n), dtype=U.dtype, device="cuda")
    H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
    F.invert(H, U, 2, z, F.Opts(alpha=1e-2, precision=F.PREC_FP64, output=F.OUT_ZETA))   # the workspace
    F.test_alloc_budget(0)
    for p in (pts, pts + 0.01):
        for k in range(4):
            F.invert(H, U, 2, out, F.Opts(alpha=1e-2, precision=F.PREC_FP64, points=p))
            assert F.test_alloc_budget(0) == (1 if k == 0 else 0)
    torch.cuda.synchronize()
    voxel = out.clone()
    F.test_alloc_budget(-1)
    for p in (pts, pts + 0.01):   # other sources ask again, and then find room for these too
        F.invert(H, U, 2, out, F.Opts(alpha=1e-2, precision=F.PREC_FP64, points=p))
    torch.cuda.synchronize()
    assert F.test_alloc_budget(-1) == 1
    tabled = torch.empty_like(out)
    F.invert(F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu), U, 2, tabled, F.Opts(alpha=1e-2, precision=F.PREC_FP64, points=pts + 0.01))
    torch.cuda.synchronize()
    assert torch.equal(out, tabled)
    assert float((out - voxel).norm()) <= 32 * torch.finfo(U.dtype).eps * float(voxel.norm())


def spectra(n, planes):
    return 8 * planes * (n // 2 + 1) * n


@pytest.mark.parametrize("n,m,mp,prec", [(192, 2, 5, 0), (192, 5, 2, 3), (256, 4, 7, 0), (384, 3, 1, 0), (512, 2, 6, 3)])
def test_plane_order_where_bin_order_finds_no_room(F, n, m, mp, prec):
    """Several observation depths: both orders project and solve the same spectra with the same kernels, so that what
    differs is the rounding of the inverse transform (FP32, a few 1e-7; 1e-5 as between the inverse's other forms)."""
    w = I.make_workload(n, mp, q=1, m_obs=m, n_incl=2, n_alpha=8, seed=73)
    U = torch.as_tensor(w.noise, dtype=torch.float32, device="cuda")
    opts = F.Opts(alpha=1e-2, output=F.OUT_ZETA, precision=prec)

    def handle():
        return F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)

    def run(H):
        out = torch.full((1, mp, n, n), float("nan"), device="cuda")
        F.invert(H, U, 1, out, opts)
        torch.cuda.synchronize()
        return out

    ref, got = run(handle()), []

    def call(budget):
        H = handle()
        F.test_alloc_budget(budget)
        got.append((run(H), H))

    b = least(F, call, spectra(n, 1) // 2, 1 << 30)
    assert b < spectra(n, 2 * max(m, mp))      # what bin order takes
    out, H = got[0]
    assert float((out - ref).norm()) <= 1e-5 * float(ref.norm())
    again = run(H)                             # the layout stays
    assert torch.equal(again, out)
    idx, res = torch.zeros(1, dtype=torch.int32, device="cuda"), {}
    for name, budget in (("plane", b), ("bin", -1)):   # the alpha rule alone, in both orders
        H2 = handle()
        F.test_alloc_budget(budget if name == "bin" else spectra(n, m) + 8 * m * (n // 2 + 1) * (n // 2 + 2) // 2 + 1024)
        res[name] = torch.zeros(8, dtype=torch.float64, device="cuda")
        F.choose_alpha(H2, U, 1, w.alphas, 0.5 * float(U.norm()), 1.1, idx, res[name], precision=prec)
        torch.cuda.synchronize()
        F.test_alloc_budget(-1)
    assert torch.equal(res["plane"], res["bin"])


def test_a_call_that_fits_in_no_order_leaves_the_handle_in_bin_order(F):
    n, m, mp = 192, 3, 6
    w = I.make_workload(n, mp, q=4, m_obs=m, n_incl=1, n_alpha=8, seed=74)
    U = torch.as_tensor(w.noise, dtype=torch.float32, device="cuda")
    out = {}
    for name in ("fresh", "after"):
        H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
        if name == "after":
            F.test_alloc_budget(spectra(n, m + mp))
            with pytest.raises(F.Fr3dError):
                F.invert(H, U, 4, torch.empty((4, mp, n, n), device="cuda"), F.Opts(alpha=1e-2, output=F.OUT_ZETA))
            F.test_alloc_budget(0)
            with pytest.raises(F.Fr3dError):
                F.choose_alpha(H, U, 4, w.alphas, 1.0, 1.1, torch.zeros(1, dtype=torch.int32, device="cuda"))
            F.test_alloc_budget(-1)
        out[name] = torch.empty((1, mp, n, n), device="cuda")
        F.invert(H, U[:1].contiguous(), 1, out[name], F.Opts(alpha=1e-2, output=F.OUT_ZETA))
        out[name + " launches"] = F.last_launch_count(H)
    torch.cuda.synchronize()
    assert out["fresh launches"] == out["after launches"]   # (plane order runs the fused inverse at this size)
    assert torch.equal(out["fresh"], out["after"])


def test_a_plan_keeps_the_queue_of_the_grids_that_find_room(F):
    """Which groups run the queue shows in their info words while the queue's counts are withheld (its bounded waits give
    up; the fused tiles of the other groups do not wait)."""
    items, refs, infos = [], [], []
    for k, (n, mp, q) in enumerate([(96, 5, 2), (256, 3, 1), (96, 2, 1), (256, 2, 2)]):
        w = I.make_workload(n, mp, q=q, n_incl=1, n_alpha=12, seed=820 + k)
        H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
        U = torch.as_tensor(w.noise, dtype=torch.float32, device="cuda")
        infos.append(torch.zeros(1, dtype=torch.int32, device="cuda"))
        opts = F.Opts(alphas=w.alphas, delta=0.3 * float(U.norm()), points=w.sources, info=infos[-1])
        items.append((H, U, q, opts, torch.empty((mp, n, n), device="cuda")))
    plan = F.Batch(items)
    F.autotune_mode(2 + 3)
    plan.run()
    torch.cuda.synchronize()
    refs = [it[4].clone() for it in items]
    plan.close()
    F.autotune_mode(2 + 5)
    large = 4 * 256 * 256 * (3 * 1 + 2 * 2) + 4096
    for budget, queued in ((1 << 30, {96, 256}), (large, {256}), (1 << 12, set())):
        F.test_alloc_budget(budget)
        plan = F.Batch(items)
        F.test_alloc_budget(-1)
        F.test_withhold_queue_counts(True)
        plan.run()
        torch.cuda.synchronize()
        F.test_withhold_queue_counts(False)
        for it, i in zip(items, infos):
            assert bool(int(i) & F.INFO_TIMEOUT) == (it[0].n in queued), (budget, it[0].n)
            it[4].fill_(float("nan"))
        plan.run()
        torch.cuda.synchronize()
        for it, ref, i in zip(items, refs, infos):
            assert torch.equal(it[4], ref) and not int(i) & F.INFO_TIMEOUT
        plan.close()


@pytest.mark.parametrize("n,m,mp,prec", [(64, 1, 6, 0), (96, 2, 5, 0), (48, 1, 16, 1), (256, 1, 9, 0)])
def test_forward_operator_one_source_at_a_time(F, n, m, mp, prec):
    """Without room for groups of sources the operator needs the planes of one source, M' + M half spectra, and a capture
    after a call with fewer sources needs no more; other sums of FP32 terms in another order (1e-5 as in the parity
    tests; FP64 1e-12)."""
    dt, tol = (torch.float64, 1e-12) if prec == F.PREC_FP64 else (torch.float32, 1e-5)
    q = 5
    w = I.make_workload(n, mp, q=1, m_obs=m, n_incl=1, seed=75)
    zeta = torch.as_tensor(np.random.default_rng(n).standard_normal((q, mp, n, n)), dtype=dt, device="cuda")

    def handle():
        return F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)

    def out():
        return torch.full((q, m, n, n), float("nan"), dtype=dt, device="cuda")

    ref, got = out(), out()
    F.fwd_apply(handle(), zeta, q, ref, prec)
    one = spectra(n, 1) * zeta.element_size() // 4
    F.test_alloc_budget((m + mp) * one + 1024)
    F.fwd_apply(handle(), zeta, q, got, prec)
    F.test_alloc_budget(-1)
    torch.cuda.synchronize()
    assert float((got - ref).norm()) <= tol * float(ref.norm())
    H, got = handle(), out()
    F.fwd_apply(H, zeta[:1].contiguous(), 1, torch.empty((1, m, n, n), dtype=dt, device="cuda"), prec)
    torch.cuda.synchronize()
    graph, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=st):
        F.fwd_apply(H, zeta, q, got, prec, stream=st)
    graph.replay()
    torch.cuda.synchronize()
    assert float((got - ref).norm()) <= tol * float(ref.norm())


@pytest.mark.parametrize("n,v", [(96, 5), (192, 5), (256, 5), (192, 4)])
def test_inverse_without_room_for_its_intermediate(F, n, v):
    """The two-pass and the queue form run the register tile instead, with the same bits; the buffer is asked for once.
    A tuner that cannot time them picks another."""
    mp, q = 6, 2
    w = I.make_workload(n, mp, q=q, n_incl=1, n_alpha=8, seed=76)
    U = torch.as_tensor(w.noise, dtype=torch.float32, device="cuda")
    opts = F.Opts(alphas=w.alphas, delta=0.3 * float(U.norm()), points=w.sources)
    zeta = torch.empty((q, mp, n, n), device="cuda")

    def handle():
        H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
        F.autotune_mode(0)
        F.invert(H, U, q, zeta, F.Opts(alphas=w.alphas, delta=0.3 * float(U.norm()), output=F.OUT_ZETA))   # the workspace
        torch.cuda.synchronize()
        return H

    ref = torch.empty((mp, n, n), device="cuda")
    H = handle()
    F.autotune_mode(2 + 3)
    F.invert(H, U, q, ref, opts)
    H = handle()
    F.autotune_mode(2 + v)
    F.test_alloc_budget(0)
    for asked in (1, 0, 0):
        out = torch.full((mp, n, n), float("nan"), device="cuda")
        F.invert(H, U, q, out, opts)
        torch.cuda.synchronize()
        assert F.test_alloc_budget(0) == asked and torch.equal(out, ref)
    F.test_alloc_budget(-1)
    H = handle()
    F.test_alloc_budget(0)
    F.autotune_mode(1)
    F.invert(H, U, q, out.fill_(float("nan")), opts)   # (a shape no other test uses: the tuner runs)
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and F.autotune_query(H)[0] < 4
