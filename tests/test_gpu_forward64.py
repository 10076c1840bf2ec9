"""The FP64 forward operator on both sides of its rule (the contraction fused with the column pass with a chunk per depth up
to eight depths, a pass of its own beyond): the launches of a call, and the result against torch's FP64 transforms of the
operator's definition (1e-12, as in the parity tests)."""
import numpy as np
import pytest

from oracle import fr3d_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mp,q,launches", [(16, 1, 1, 4), (48, 8, 1, 4), (48, 9, 2, 5), (192, 6, 1, 4), (192, 8, 3, 4),
                                             (192, 9, 1, 5), (256, 64, 1, 5), (512, 3, 1, 4)])
def test_fp64_forward_operator(n, mp, q, launches):
    from paper_1703_01216_gb300 import fr3d as F
    rng = np.random.default_rng(n + mp)
    h = 2.0 / n
    zr, nu = 0.5 + (np.arange(mp) + 0.5) * 0.5 / mp, np.full(mp, 0.5 / mp)
    zeta = torch.tensor(rng.standard_normal((q, mp, n, n)), device="cuda")
    lag = torch.tensor(O.wrapped_lags(n) * h, device="cuda")
    Z, acc = torch.fft.rfft2(zeta), 0
    for j in range(mp):
        dz = float(-zr[j])
        r2 = lag[None, :] ** 2 + lag[:, None] ** 2 + dz * dz
        acc = acc + h * h * nu[j] * torch.fft.rfft2(-dz / (r2 * torch.sqrt(r2))).real * Z[:, j]
    ref = torch.fft.irfft2(acc, s=(n, n))[:, None]
    H = F.kernel_transform(n, -1.0, h, zr, np.zeros(1), nu)
    U = torch.full((q, 1, n, n), float("nan"), dtype=torch.float64, device="cuda")
    F.fwd_apply(H, zeta, q, U, F.PREC_FP64)
    torch.cuda.synchronize()
    assert float((U - ref).norm() / ref.norm()) <= 1e-12
    assert F.last_launch_count(H) == launches
