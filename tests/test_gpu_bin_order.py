"""Spectra of several observation depths in bin order (records of Q M values per frequency, n >= 192) against the
FP64 oracle, on both sides of the rule's line: odd numbers of observation and result depths (ragged plane groups of
the column passes), fewer and more result than observation depths, both outputs, both product precisions.

Tolerance: 1e-4 relative at alpha = 1e-3, the bound of the plane-ordered path at alpha >= 1e-4 (FP32 data spectra,
projected components and solve tables, or the hi + lo form that is held to the same bound; amplified by at most
1/(2 sqrt(alpha))).
"""

import numpy as np
import pytest

import oracle as O
from paper_1703_01216_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


@pytest.mark.parametrize("n,mp,q,m", [(128, 3, 1, 2), (192, 7, 1, 3), (192, 2, 3, 5), (256, 3, 2, 3)])
def test_bin_order_matches_oracle(n, mp, q, m):
    from paper_1703_01216_gb300 import build, fr3d as F
    build.build()
    w = I.make_workload(n, mp, q=q, m_obs=m, n_incl=3, noise_level=0.02, n_alpha=8, seed=1300 + n + m)
    A = O.A_matrices(n, w.h, w.zy, w.zr, w.nu)
    U = O.forward_dft(O.zeta_from_xi(w.xi_true, w.sources, n, w.x0, w.h, w.zr), n, w.h, w.zy, w.zr, w.nu, A=A) + w.noise
    H = F.kernel_transform(n, w.x0, w.h, w.zr, w.zy, w.nu)
    for kind, name, shape in ((F.OUT_XI, "xi", (mp, n, n)), (F.OUT_ZETA, "zeta", (q, mp, n, n))):
        ref = O.invert(U, n, w.x0, w.h, w.zy, w.zr, w.nu, alpha=1e-3, sources=w.sources, A=A, output=name)[name]
        for prec in (F.PREC_FP32, F.PREC_BF16X3):
            o = torch.full(shape, float("nan"), device="cuda")
            F.invert(H, dev(U), q, o, F.Opts(alpha=1e-3, output=kind, points=w.sources, precision=prec))
            torch.cuda.synchronize()
            assert rel(o.double().cpu().numpy(), ref) <= 1e-4, (name, prec)
