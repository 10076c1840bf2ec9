"""The combination with tabled weights (the default) against the per-voxel evaluation of V0 (taken when the
table cannot be built, here: a first xi call inside a stream capture)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1703_01216_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mp,q,prec", [(16, 1, 1, 1), (24, 5, 3, 1), (48, 7, 2, 1), (512, 2, 2, 0)])
def test_tabled_weights_match_the_per_voxel_combination(n, mp, q, prec):
    from paper_1703_01216_gb300 import fr3d as F
    w = I.make_workload(n, mp, q=q, n_incl=1, seed=61)
    dt = torch.float64 if prec == F.PREC_FP64 else torch.float32
    U = torch.as_tensor(w.noise, dtype=dt, device="cuda")
    H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
    xi = torch.empty((mp, n, n), dtype=dt, device="cuda")
    zeta = torch.empty((q, mp, n, n), dtype=dt, device="cuda")
    # everything but the table: workspace and fixed-level table (a zeta call), the sources (zeta_from_xi)
    F.invert(H, U, q, zeta, F.Opts(alpha=1e-2, output=F.OUT_ZETA, precision=prec))
    F.zeta_from_xi(H, torch.ones_like(xi), w.sources, torch.empty_like(zeta), precision=prec)
    opts = F.Opts(alpha=1e-2, precision=prec, points=w.sources)
    g = torch.cuda.CUDAGraph()
    st = torch.cuda.Stream()
    with torch.cuda.graph(g, stream=st):
        F.invert(H, U, q, xi, opts, stream=st)
    g.replay()
    torch.cuda.synchronize()
    direct = xi.clone()
    F.invert(H, U, q, xi, opts)
    torch.cuda.synchronize()
    a, b = direct.double().cpu().numpy(), xi.double().cpu().numpy()
    assert np.isfinite(a).all() and np.linalg.norm(b) > 0
    # both combine the same zeta; the weights differ by their rounding (a few ulp of the precision per voxel)
    assert np.linalg.norm(a - b) <= 32 * torch.finfo(dt).eps * np.linalg.norm(b)
