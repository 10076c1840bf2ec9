"""Residual sums of the discrepancy rule at several observation depths: the per-band curves of the same data add up
to the one-band curve (every class's FP32 contribution is the same; only the order of FP64 sums differs: 1e-12),
at candidate and band counts around the finishing block's 1024 threads."""
import numpy as np
import pytest

from paper_1703_01216_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nb,na", [(16, 2, 1), (32, 7, 33), (48, 16, 64), (64, 9, 128), (32, 16, 128)])
def test_band_curves_add_up(n, nb, na):
    from paper_1703_01216_gb300 import fr3d as F
    w = I.make_workload(n, 5, q=2, m_obs=3, n_incl=2, seed=n + nb, n_alpha=na)
    U = torch.as_tensor(w.noise, dtype=torch.float32, device="cuda")
    H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
    xi = torch.empty((w.Mp, n, n), device="cuda")
    curves = {}
    for b in (1, nb):
        idx = torch.zeros(b, dtype=torch.int32, device="cuda")
        res = torch.full((b, na), float("nan"), dtype=torch.float64, device="cuda")
        F.invert(H, U, w.Q, xi, F.Opts(alphas=w.alphas, delta=float(U.norm()), points=w.sources, alpha_idx=idx,
                                       residuals=res, n_bands=b))
        torch.cuda.synchronize()
        curves[b] = res.cpu().numpy()
    assert np.isfinite(curves[nb]).all() and (curves[1] > 0).all()
    assert np.max(np.abs(curves[nb].sum(0) - curves[1][0]) / curves[1][0]) <= 1e-12
