"""The alpha rule at the grid sizes where its block and group counts change (8 to 64 classes per block, one or two
levels of tickets, the last block short), for few and many planes, candidates and bands: residual curves against an
FP64 evaluation of the rule's formula from torch's transforms.  The class powers are FP32 sums of at most 4 Q
squares of FP32 spectra (relative 4 Q 2^-24 plus the spectrum's own 1e-7 per bin, averaged over thousands: 1e-5 as in
the parity tests); FP64 mode 1e-11."""
import numpy as np
import pytest

from oracle import fr3d_oracle as O
from paper_1703_01216_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,q,na,nb", [(16, 1, 1, 1), (24, 3, 7, 1), (32, 1, 16, 1), (64, 2, 33, 5), (96, 5, 32, 1),
                                       (128, 1, 128, 16), (192, 9, 64, 8), (256, 8, 64, 1), (384, 2, 17, 1),
                                       (512, 1, 40, 3)])
def test_residual_curves(n, q, na, nb):
    from paper_1703_01216_gb300 import fr3d as F
    mp = 3
    w = I.make_workload(n, mp, q=q, n_incl=1, n_alpha=na, seed=n + q)
    U = torch.as_tensor(w.noise, dtype=torch.float32, device="cuda")
    lag = torch.tensor(O.wrapped_lags(n) * w.h, device="cuda")
    nrm = 0
    for j in range(mp):
        dz = float(w.zy[0] - w.zr[j])
        r2 = lag[None, :] ** 2 + lag[:, None] ** 2 + dz * dz
        a = w.h * w.h * float(w.nu[j]) * torch.fft.fft2(-dz / (r2 * torch.sqrt(r2))).real
        nrm = nrm + a * a
    s2 = float(nrm.max())
    P = torch.fft.fft2(U[:, 0].double()).abs().square().sum(0)
    band = torch.tensor(O.radial_bands(n, nb).reshape(n, n), device="cuda")
    ref = torch.empty((nb, na), dtype=torch.float64)
    for k, al in enumerate(w.alphas):
        r = (float(al) * s2 / (nrm + float(al) * s2)) ** 2 * P / (n * n)
        for b in range(nb):
            ref[b, k] = r[band == b].sum()
    H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
    for prec, dt, tol in ((F.PREC_FP32, torch.float32, 1e-5), (F.PREC_FP64, torch.float64, 1e-11)):
        xi = torch.empty((mp, n, n), dtype=dt, device="cuda")
        for rep in range(2):    # the tickets are left at zero
            res = torch.full((nb, na), float("nan"), dtype=torch.float64, device="cuda")
            idx = torch.full((nb,), -1, dtype=torch.int32, device="cuda")
            F.invert(H, U.to(dt), q, xi, F.Opts(alphas=w.alphas, delta=0.5 * float(U.norm()), points=w.sources,
                                                residuals=res, alpha_idx=idx, n_bands=nb, precision=prec))
            torch.cuda.synchronize()
            got = res.cpu()
            assert float(((got - ref).abs() / ref).max()) <= tol
            assert int(idx.min()) >= 0
