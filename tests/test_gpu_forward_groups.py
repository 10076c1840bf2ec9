"""The forward operator with its sources in groups and its depths in chunks against FP64 (torch's FFTs of the
operator's definition): one depth, depths that leave a short chunk, single- and three-pass transform lengths, several
sources, several observation depths.  Tolerances: FP32 transforms and sums, 1e-6 per pass of a few ulp each (1e-5 as
in the parity tests); FP64 1e-12."""
import numpy as np
import pytest

from oracle import fr3d_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mp,m,q", [(16, 1, 1, 1), (16, 9, 1, 3), (24, 5, 1, 2), (96, 33, 1, 3), (128, 7, 1, 1),
                                      (192, 13, 1, 2), (256, 70, 1, 5), (384, 6, 1, 2), (512, 5, 1, 3), (48, 6, 2, 4)])
def test_forward_groups_and_chunks(n, mp, m, q):
    from paper_1703_01216_gb300 import fr3d as F
    rng = np.random.default_rng(n + mp)
    h, x0 = 2.0 / n, -1.0
    zr, nu = 0.5 + (np.arange(mp) + 0.5) * 0.5 / mp, np.full(mp, 0.5 / mp)
    zy = -0.1 * np.arange(m)
    zeta = torch.tensor(rng.standard_normal((q, mp, n, n)), device="cuda")
    lag = torch.tensor(O.wrapped_lags(n) * h, device="cuda")
    Z = torch.fft.rfft2(zeta)
    ref = torch.empty((q, m, n, n), dtype=torch.float64, device="cuda")
    for i in range(m):
        acc = 0
        for j in range(mp):
            dz = float(zy[i] - zr[j])
            r2 = lag[None, :] ** 2 + lag[:, None] ** 2 + dz * dz
            acc = acc + h * h * nu[j] * torch.fft.rfft2(-dz / (r2 * torch.sqrt(r2))).real * Z[:, j]
        ref[:, i] = torch.fft.irfft2(acc, s=(n, n))
    H = F.kernel_transform(n, x0, h, zr, zy, nu)
    for prec, dt, tol in ((F.PREC_FP32, torch.float32, 1e-5), (F.PREC_FP64, torch.float64, 1e-12)):
        U = torch.full((q, m, n, n), float("nan"), dtype=dt, device="cuda")
        F.fwd_apply(H, zeta.to(dt), q, U, prec)
        torch.cuda.synchronize()
        assert float((U.double() - ref).norm() / ref.norm()) <= tol
