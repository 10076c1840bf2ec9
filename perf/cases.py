"""Performance cases of the library: what users have it do, through the public binding.

A case is a dict of plain values.  `listed()` names the standing cases, `draw(rng)` gives one more from the same
ranges, `prepare(case, seed)` makes what a program holds before the call (handle, data, options, output buffers),
`run(state)` is one call as a program makes it, `work(case)` the bytes and operations no implementation can do
without, `exact(case, seed)` the result in 64 bits from torch alone.

Data are synthetic: seeded Gaussian and ellipsoidal inclusions, the spectral forward model evaluated in FP64 by
torch, relative Gaussian noise of 0.5-5 % (the benchmark configurations' range), one observation plane unless
stated.
"""

from __future__ import annotations

import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_1703_01216_gb300 import fr3d, inputs
from paper_1703_01216_gb300.synth import PhantomSampler

TAU = 1.1
UNET_WIDTHS = (16, 32, 64, 128)


# --------------------------------------------------------------------------------------------- the cases
def _invert(name, n, depths, sources, alphas, noise, *, planes=1, bands=1, precision="fp32", ra="tikhonov",
            output="xi", pad=1, where="device"):
    return {"name": name, "kind": "invert", "n": n, "depths": depths, "planes": planes, "sources": sources,
            "alphas": alphas, "noise": noise, "bands": bands, "precision": precision, "ra": ra, "output": output,
            "pad": pad, "where": where}


def listed():
    return [
        # one small problem in the paper's own arithmetic: the smallest call, a script trying the method out
        _invert("small_fp64", 32, 16, 1, 16, 0.01, precision="fp64"),
        # an ordinary single-source reconstruction, as the training pairs of the post-corrector are made
        _invert("plain_128", 128, 32, 1, 32, 0.02),
        # the headline workload: 8 source parameters sharing one unknown, 64 candidate alphas
        _invert("sources_256", 256, 64, 8, 64, 0.01),
        # a radix-3 grid with an odd depth and source count, one alpha per radial band
        _invert("bands_192", 192, 51, 5, 32, 0.03, bands=8),
        # the headline workload in the paper's arithmetic (a reference reconstruction)
        _invert("sources_256_fp64", 256, 64, 8, 64, 0.01, precision="fp64"),
        # the headline workload from and to page-locked host memory (a program without device buffers)
        _invert("sources_256_host", 256, 64, 8, 64, 0.01, where="host"),
        # the paper's experiment: 51 observation and 51 unknown depths at 512^2, truncated SVD
        _invert("paper_512", 512, 51, 1, 32, 0.01, planes=51, ra="tsvd"),
        # several observation depths with the products on the tensor cores in split BF16
        _invert("planes_256_bf16x3", 256, 64, 1, 32, 0.01, planes=40, precision="bf16x3"),
        # a serving queue: 64 independent instances of uneven grid, depth and source counts in one plan
        {"name": "batch_64", "kind": "batch", "count": 64, "shapes": 4000},
        # the forward operator on all sources (simulating data, making training pairs)
        {"name": "forward_256", "kind": "forward", "n": 256, "depths": 64, "planes": 1, "sources": 8,
         "precision": "fp32"},
        # post-correcting a batch of reconstructions, and one training gradient of the same batch
        {"name": "unet_forward", "kind": "unet", "depth": 32, "height": 128, "width": 128, "batch": 8,
         "what": "forward"},
        {"name": "unet_gradient", "kind": "unet", "depth": 32, "height": 128, "width": 128, "batch": 8,
         "what": "gradient"},
    ]


def _between(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["invert", "invert", "invert", "fp64", "planes", "batch", "forward", "unet", "unet"])
    if kind == "batch":
        return {"kind": "batch", "count": _between(rng, 5, 60), "shapes": rng.randrange(1 << 20)}
    if kind == "unet":
        d, h, w = 8 * _between(rng, 1, 5), 8 * _between(rng, 3, 20), 8 * _between(rng, 3, 20)
        return {"kind": "unet", "depth": d, "height": h, "width": w,
                "batch": max(1, min(rng.randint(1, 8), (8 * 32 * 128 * 128) // (d * h * w))),
                "what": rng.choice(["forward", "gradient"])}
    if kind == "planes":
        n = rng.choice([32, 48, 64, 96, 128, 192, 256])
        c = _invert("", n, _between(rng, 6, 64), rng.choice([1, 1, 2]), rng.choice([16, 32]), rng.uniform(0.005, 0.05),
                    planes=_between(rng, 3, 56), precision=rng.choice(["fp32", "fp32", "bf16x3"]),
                    ra=rng.choice(["tikhonov", "tsvd"]))
    elif kind == "fp64":
        c = _invert("", rng.choice([32, 48, 64, 96, 128, 192]), _between(rng, 8, 64), rng.randint(1, 6),
                    rng.choice([16, 32, 64]), rng.uniform(0.005, 0.05), precision="fp64",
                    output=rng.choice(["xi", "xi", "zeta"]))
    elif kind == "forward":
        c = {"kind": "forward", "n": rng.choice([48, 64, 96, 128, 192, 256, 384]), "depths": _between(rng, 8, 64),
             "planes": rng.choice([1, 1, 1, 4]), "sources": rng.randint(1, 8), "precision": "fp32"}
    else:
        n = rng.choice([32, 64, 96, 128, 192, 256, 256, 384, 512])
        c = _invert("", n, _between(rng, 8, 64), rng.randint(1, 8), rng.choice([16, 32, 64]), rng.uniform(0.005, 0.05),
                    bands=rng.choice([1, 1, 1, 8]), ra=rng.choice(["tikhonov", "tikhonov", "tsvd"]),
                    output=rng.choice(["xi", "xi", "xi", "zeta"]),
                    pad=rng.choice([1, 1, 1, 2]) if n <= 128 else 1, where=rng.choice(["device", "device", "host"]))
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------- geometry and the 64-bit model
def _dev():
    return torch.device("cuda")


def _geometry(case):
    """Grid, depths, weights, observation depths, source points and candidates of one inversion or forward case."""
    n, m = case["n"], case.get("planes", 1)
    g = {"n": n, "M": m, "Mp": case["depths"], "Q": case["sources"], "pad": case.get("pad", 1)}
    if m > 1:  # the paper's experiment: R = [-10, 10]^2 x [1, 2], Y the same square x [6, 7], its ten point sources
        g["h"], g["x0"], g["scale"] = 20.0 / n, -10.0, 10.0
        g["zr"], g["nu"] = inputs.slab_depths(g["Mp"], 1.0, 2.0)
        g["zy"] = inputs.slab_depths(m, 6.0, 7.0)[0]
        cross = inputs.cross_sources(g["Q"], offset=8.0, z_step=0.0)
        g["points"] = np.concatenate([cross, cross], axis=1)
        for q in range(g["Q"]):
            g["points"][q, :5, 2], g["points"][q, 5:, 2] = 3.0 + 0.2 * q, 5.0 + 0.2 * q
    else:      # the synthetic slab of the benchmark configurations
        g["h"], g["x0"], g["scale"] = 2.0 / n, -1.0, 1.0
        g["zr"], g["nu"] = inputs.slab_depths(g["Mp"])
        g["zy"] = np.zeros(1)
        g["points"] = inputs.cross_sources(g["Q"])
    if "alphas" in case:
        g["alphas"] = np.logspace(-8.0, -1.0, case["alphas"])
    return g


def _kernel_spectra(g):
    """A^(m) of Eq. (6) on the half spectrum, [M, M', L, L/2 + 1] in FP64 (the sampled kernel's DFT is real)."""
    L = g["pad"] * g["n"]
    t = torch.arange(L, device=_dev(), dtype=torch.float64)
    lag = torch.where(t < L // 2, t, t - L) * g["h"]
    rho2 = lag[None, :] ** 2 + lag[:, None] ** 2
    zr = torch.tensor(g["zr"], device=_dev())
    A = torch.empty((g["M"], g["Mp"], L, L // 2 + 1), device=_dev(), dtype=torch.float64)
    for i, zy in enumerate(g["zy"]):
        dz = (float(zy) - zr)[:, None, None]
        r2 = rho2 + dz * dz
        K = -dz / (r2 * torch.sqrt(r2))
        A[i] = torch.fft.rfft2(K).real * (g["h"] ** 2) * torch.tensor(g["nu"], device=_dev())[:, None, None]
    return A


def _v0(g):
    """V0_q on the grid of R, [Q, M', n, n] in FP64."""
    c = torch.tensor(g["x0"] + (np.arange(g["n"]) + 0.5) * g["h"], device=_dev())
    z = torch.tensor(g["zr"], device=_dev())[:, None, None]
    out = torch.zeros((g["Q"], g["Mp"], g["n"], g["n"]), device=_dev(), dtype=torch.float64)
    for q in range(g["Q"]):
        for x, y, zl in g["points"][q]:
            out[q] += torch.rsqrt((c[None, None, :] - x) ** 2 + (c[None, :, None] - y) ** 2 + (z - zl) ** 2)
    return out.mul_(-1.0 / (4.0 * math.pi))


def _pad(f, g):
    L = g["pad"] * g["n"]
    return torch.nn.functional.pad(f, (0, L - g["n"], 0, L - g["n"]))


def _forward(zeta, A, g):
    """U_q = A zeta_q, [Q, M, n, n] in FP64."""
    L, n = g["pad"] * g["n"], g["n"]
    U = torch.empty((zeta.shape[0], g["M"], n, n), device=_dev(), dtype=torch.float64)
    for q in range(zeta.shape[0]):
        Z = torch.fft.rfft2(_pad(zeta[q].double(), g))
        for i in range(g["M"]):
            U[q, i] = torch.fft.irfft2((A[i] * Z).sum(0), s=(L, L))[:n, :n]
    return U


def _phantom(g, seed, n_incl=(1, 12)):
    s = g["scale"]
    rng = np.random.default_rng(seed)
    sampler = PhantomSampler(g["n"], g["x0"], g["h"], g["zr"], _dev(), width=(0.1 * s, 0.2 * s), semi=(0.1 * s, 0.3 * s))
    return sampler.draw(rng, int(rng.integers(n_incl[0], n_incl[1] + 1))).double()


def _data(g, noise, seed, A=None):
    """Noisy data U [Q, M, n, n] (FP64 on the device) of a seeded phantom, and the norm of the noise."""
    A = _kernel_spectra(g) if A is None else A
    U = _forward(_phantom(g, seed)[None] * _v0(g), A, g)
    gen = torch.Generator(device=_dev())
    gen.manual_seed(seed)
    e = torch.randn(U.shape, generator=gen, device=_dev(), dtype=torch.float32).double()
    e *= noise * U.norm() / e.norm()
    return U + e, float(e.norm())


def _band_map(L, bands):
    """Radial band of every half-spectrum bin, and the share of the whole spectrum's bins in each band."""
    k = np.arange(L)
    kf = np.minimum(k, L - k)
    full = np.minimum(np.floor(bands * np.sqrt(kf[None, :] ** 2 + kf[:, None] ** 2) / (math.sqrt(2.0) * (L // 2))),
                      bands - 1).astype(np.int64)
    share = np.bincount(full.ravel(), minlength=bands) / (L * L)
    return torch.tensor(full[:, :L // 2 + 1], device=_dev()), share


def _choose(r2, bound):
    ok = np.nonzero(r2 <= bound ** 2)[0]
    return int(ok.max()) if ok.size else 0


def _solve_planes(A, Uh, g, alphas, delta, ra):
    """Several observation depths: spectra of zeta [Q, M', L, L/2 + 1] and the chosen index, through the
    eigendecomposition of A A^T per frequency class (the 8 symmetric frequencies share one matrix)."""
    L = g["pad"] * g["n"]
    s2 = float((A * A).sum((0, 1)).max())
    half = L // 2 + 1
    ky = torch.arange(L, device=_dev())
    v = torch.minimum(ky, L - ky)[:, None].expand(L, half)
    u = torch.arange(half, device=_dev())[None, :].expand(L, half)
    cls = (torch.maximum(u, v) * (torch.maximum(u, v) + 1) // 2 + torch.minimum(u, v)).reshape(-1)
    C = half * (half + 1) // 2
    first = torch.full((C,), L * half, device=_dev(), dtype=torch.int64)
    first.scatter_reduce_(0, cls, torch.arange(L * half, device=_dev()), "amin")
    Ac = A.reshape(g["M"], g["Mp"], -1)[:, :, first].permute(2, 0, 1).contiguous()
    gram = (Ac @ Ac.transpose(1, 2)).cpu().numpy()
    with ThreadPoolExecutor(16) as pool:
        parts = list(pool.map(np.linalg.eigh, np.array_split(gram, min(64, C))))
    lam = torch.tensor(np.concatenate([p[0] for p in parts]), device=_dev()).clamp_(min=0)
    V = torch.tensor(np.concatenate([p[1] for p in parts]), device=_dev())
    wt = torch.full((L, half), 2.0, device=_dev(), dtype=torch.float64)
    wt[:, 0] = wt[:, -1] = 1.0
    D = torch.view_as_real(Uh.reshape(g["Q"], g["M"], -1)).permute(2, 1, 0, 3).reshape(L * half, g["M"], -1)
    P = torch.zeros((C, g["M"]), device=_dev(), dtype=torch.float64)
    step = 16384
    for b in range(0, L * half, step):
        c = cls[b:b + step]
        p = V[c].transpose(1, 2) @ D[b:b + step]
        P.index_add_(0, c, p.square().sum(2) * wt.reshape(-1)[b:b + step, None])
    def left(a):  # squared residual at candidate a
        f = (lam < a * s2).double() if ra == "tsvd" else (a * s2 / (lam + a * s2)) ** 2
        return float((f * P).sum()) / (L * L)
    k = _choose(np.array([left(float(a)) for a in alphas]), TAU * delta)
    t = float(alphas[k]) * s2
    w = torch.where(lam >= t, 1.0 / lam.clamp(min=1e-300), 0.0) if ra == "tsvd" else 1.0 / (lam + t)
    S = Ac.transpose(1, 2) @ (V * w[:, None, :]) @ V.transpose(1, 2)
    Z = torch.empty((L * half, g["Mp"], 2 * g["Q"]), device=_dev(), dtype=torch.float64)
    for b in range(0, L * half, step):
        Z[b:b + step] = S[cls[b:b + step]] @ D[b:b + step]
    Z = torch.view_as_complex(Z.reshape(L * half, g["Mp"], g["Q"], 2).contiguous())
    return Z.permute(2, 1, 0).reshape(g["Q"], g["Mp"], L, half), [k]


def _solve_plane(A, Uh, g, alphas, delta, ra, bands):
    """One observation depth: the same, in closed form."""
    L = g["pad"] * g["n"]
    a = A[0]
    nrm = (a * a).sum(0)
    s2 = float(nrm.max())
    P = (Uh[:, 0].real ** 2 + Uh[:, 0].imag ** 2).sum(0)
    P[:, 1:-1] *= 2.0
    band, share = _band_map(L, bands)
    ks, weight = [], torch.empty_like(nrm)
    for b in range(bands):
        at = band == b
        nb, pb = nrm[at], P[at]
        def left(al):
            f = (nb < al * s2).double() if ra == "tsvd" else (al * s2 / (nb + al * s2)) ** 2
            return float((f * pb).sum()) / (L * L)
        bound = TAU * delta * (math.sqrt(share[b]) if bands > 1 else 1.0)
        k = _choose(np.array([left(float(al)) for al in alphas]), bound)
        t = float(alphas[k]) * s2
        weight[at] = torch.where(nb >= t, 1.0 / nb, 0.0) if ra == "tsvd" else 1.0 / (nb + t)
        ks.append(k)
    return (a[None] * weight) * Uh, ks


def _invert_exact(U, g, A, alphas, delta, ra="tikhonov", bands=1, output="xi"):
    L, n = g["pad"] * g["n"], g["n"]
    Uh = torch.fft.rfft2(_pad(U.double(), g))
    if g["M"] > 1:
        Z, ks = _solve_planes(A, Uh, g, alphas, delta, ra)
    else:
        Z, ks = _solve_plane(A, Uh, g, alphas, delta, ra, bands)
    zeta = torch.empty((g["Q"], g["Mp"], n, n), device=_dev(), dtype=torch.float64)
    for q in range(g["Q"]):
        zeta[q] = torch.fft.irfft2(Z[q], s=(L, L))[:, :n, :n]
    if output == "zeta":
        return zeta, ks
    v = _v0(g)
    return (v * zeta).sum(0) / (v * v).sum(0), ks


# ------------------------------------------------------------------------------------------- the kinds of case
PRECISION = {"fp32": fr3d.PREC_FP32, "fp64": fr3d.PREC_FP64, "bf16x3": fr3d.PREC_BF16X3}


def _handle(g):
    return fr3d.kernel_transform(g["n"], g["x0"], g["h"], g["zr"], g["zy"], g["nu"], pad=g["pad"])


def _invert_inputs(case, seed):
    g = _geometry(case)
    A = _kernel_spectra(g)
    U, delta = _data(g, case["noise"], seed, A)
    if case["precision"] != "fp64":
        U = U.float()
    return g, A, U, delta


def _prepare_invert(case, seed):
    g, _, U, delta = _invert_inputs(case, seed)
    shape = (g["Mp"], g["n"], g["n"]) if case["output"] == "xi" else (g["Q"], g["Mp"], g["n"], g["n"])
    idx = torch.zeros(case["bands"], dtype=torch.int32, device=_dev())
    opts = fr3d.Opts(alphas=g["alphas"], delta=delta, tau=TAU, points=g["points"], alpha_idx=idx,
                     n_bands=case["bands"], precision=PRECISION[case["precision"]],
                     ra=fr3d.RA_TSVD if case["ra"] == "tsvd" else fr3d.RA_TIKHONOV,
                     output=fr3d.OUT_XI if case["output"] == "xi" else fr3d.OUT_ZETA)
    if case["where"] == "host":
        U = U.cpu().pin_memory()
        out = torch.empty(shape, dtype=U.dtype).pin_memory()
        call = fr3d.invert_host
    else:
        out = torch.empty(shape, dtype=U.dtype, device=_dev())
        call = fr3d.invert
    return {"call": call, "handle": _handle(g), "U": U.contiguous(), "Q": g["Q"], "out": out, "opts": opts, "idx": idx}


def _batch_shapes(case):
    rng = np.random.default_rng(case["shapes"])
    got = []
    for _ in range(case["count"]):
        c = {"n": int(rng.choice([64, 96, 128, 192, 256])), "depths": int(rng.choice([16, 32, 48, 64])),
             "sources": int(rng.integers(1, 9)), "alphas": 32}
        rng.integers(1, 11)  # (inclusion count: drawn with the phantom)
        c["noise"] = float(rng.uniform(0.005, 0.05))
        got.append(c)
    return got


def _prepare_batch(case, seed):
    items = []
    for k, c in enumerate(_batch_shapes(case)):
        g = _geometry(c)
        U, delta = _data(g, c["noise"], seed * 1000 + k)
        out = torch.empty((g["Mp"], g["n"], g["n"]), device=_dev())
        items.append((_handle(g), U.float().contiguous(), g["Q"],
                      fr3d.Opts(alphas=g["alphas"], delta=delta, tau=TAU, points=g["points"]), out))
    return {"plan": fr3d.Batch(items), "outs": [it[4] for it in items], "items": items}


def _forward_inputs(case, seed):
    g = _geometry(case)
    zeta = _phantom(g, seed)[None] * _v0(g)
    return g, zeta.double() if case["precision"] == "fp64" else zeta.float()


def _prepare_forward(case, seed):
    g, zeta = _forward_inputs(case, seed)
    U = torch.empty((g["Q"], g["M"], g["n"], g["n"]), dtype=zeta.dtype, device=_dev())
    return {"handle": _handle(g), "zeta": zeta, "Q": g["Q"], "U": U, "precision": PRECISION[case["precision"]]}


def _unet_specs():
    """(c_in, c_out, level) of the 15 convolutions in parameter order."""
    w = UNET_WIDTHS
    s = [(1, w[0], 0), (w[0], w[0], 0)]
    for l in (1, 2):
        s += [(w[l - 1], w[l], l), (w[l], w[l], l)]
    s += [(w[2], w[3], 3), (w[3], w[3], 3), (w[3], w[3], 3)]
    for l in (2, 1, 0):
        s += [(w[l + 1] + w[l], w[l], l), (w[l], w[l], l)]
    return s


def _unet_params(seed):
    """He-normal weights, small biases and a small head: a network part way through training."""
    rng = np.random.default_rng(seed)
    p = []
    for ci, co, _ in _unet_specs():
        p += [rng.standard_normal(co * ci * 27) * math.sqrt(2.0 / (27 * ci)), 0.02 * rng.standard_normal(co)]
    p += [0.1 * rng.standard_normal(UNET_WIDTHS[0]), 0.02 * rng.standard_normal(1)]
    return np.concatenate(p).astype(np.float32)


def _unet_inputs(case, seed):
    """Plain reconstructions x (FP32) of noisy data and the true volumes t."""
    d, h, w, b = case["depth"], case["height"], case["width"], case["batch"]
    n = 16
    while n < max(h, w):
        n = n * 3 // 2 if n & (n - 1) == 0 else n * 4 // 3
    g = _geometry({"n": n, "depths": d, "sources": 1, "alphas": 32})
    A, v = _kernel_spectra(g), _v0(g)
    x = torch.empty((b, d, h, w), device=_dev())
    t = torch.empty_like(x)
    for k in range(b):
        xi = _phantom(g, seed * 100 + k)
        U, delta = _data(g, 0.02, seed * 100 + k, A)
        a = A[0]
        nrm = (a * a).sum(0)
        Z = a * (torch.fft.rfft2(U[0, 0]) / (nrm + 1e-3 * nrm.max()))
        x[k] = (torch.fft.irfft2(Z, s=(n, n)) / v[0])[:, :h, :w].float()
        t[k] = xi[:, :h, :w].float()
    return x, t


def _prepare_unet(case, seed):
    x, t = _unet_inputs(case, seed)
    net = fr3d.Unet(case["depth"], case["height"], case["width"], case["batch"], 4.0, seed & 0xFFFF)
    net.set_params(_unet_params(seed))
    s = {"net": net, "x": x, "t": t, "y": torch.empty_like(x), "loss": torch.zeros(1, device=_dev())}
    if case["what"] == "gradient":
        s["grad"] = torch.zeros(net.n_params, device=_dev())
    return s


def _lrelu(z):
    return torch.where(z > 0, z, 0.01 * z)


def _conv64(x, w, b):
    """3 x 3 x 3 zero-padded correlation as 27 shifted products; x [ci, D, H, W]."""
    _, D, H, W = x.shape
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    out = b[:, None]
    for a in range(3):
        for e in range(3):
            for f in range(3):
                out = out + w[:, :, a, e, f] @ xp[:, a:a + D, e:e + H, f:f + W].reshape(x.shape[0], -1)
    return out.reshape(-1, D, H, W)


def _unet_exact(x, p, in_scale):
    """The network in FP64 on one volume x [D, H, W]: prediction in scaled units."""
    specs, at, layers = _unet_specs(), 0, []
    for ci, co, _ in specs:
        layers.append((p[at:at + co * ci * 27].reshape(co, ci, 3, 3, 3), p[at + co * ci * 27:at + co * ci * 27 + co]))
        at += co * ci * 27 + co
    def conv(k, z):
        return _lrelu(_conv64(z, *layers[k]))
    def pool(z):
        return torch.nn.functional.avg_pool3d(z[None], 2)[0]
    def up(z):
        return z.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)
    xs = in_scale * x
    z, skips = conv(1, conv(0, xs[None])), []
    for l in (1, 2):
        skips.append(z)
        z = conv(2 * l + 1, conv(2 * l, pool(z)))
    skips.append(z)
    z = conv(8, conv(7, conv(6, pool(z))))
    for k, l in ((9, 2), (11, 1), (13, 0)):
        z = conv(k + 1, conv(k, torch.cat([up(z), skips[l]])))
    return xs + (p[at:at + UNET_WIDTHS[0]] @ z.reshape(UNET_WIDTHS[0], -1)).reshape(x.shape) + p[at + UNET_WIDTHS[0]]


# ------------------------------------------------------------------------------------------------- the interface
def prepare(case, seed):
    kind = case["kind"]
    state = {"invert": _prepare_invert, "batch": _prepare_batch, "forward": _prepare_forward,
             "unet": _prepare_unet}[kind](case, seed)
    state["kind"] = kind
    return state


def run(state):
    kind = state["kind"]
    if kind == "invert":
        state["call"](state["handle"], state["U"], state["Q"], state["out"], state["opts"])
        return {"out": state["out"], "alpha_idx": state["idx"]}
    if kind == "batch":
        state["plan"].run()
        return state["outs"]
    if kind == "forward":
        fr3d.fwd_apply(state["handle"], state["zeta"], state["Q"], state["U"], state["precision"])
        return state["U"]
    if "grad" in state:
        state["net"].gradient(state["x"], state["t"], state["grad"], state["loss"])
        return {"grad": state["grad"], "loss": state["loss"]}
    state["net"].forward(state["x"], state["y"])
    return state["y"]


def _fft_flops(L):
    """One real 2D transform of L x L points: half of the complex count 5 N log2 N."""
    return 2.5 * L * L * math.log2(L * L)


def _work_invert(c):
    n, m, mp, q = c["n"], c.get("planes", 1), c["depths"], c["sources"]
    el = 8 if c.get("precision") == "fp64" else 4
    L = c.get("pad", 1) * n
    bins, classes = L * (L // 2 + 1), (L // 2 + 1) * (L // 2 + 2) // 2
    xi = c.get("output", "xi") == "xi"
    # data, result, and the kernel's table (one entry per frequency class, observation and unknown depth)
    by = el * (q * m * n * n + (1 if xi else q) * mp * n * n + classes * m * mp)
    fl = q * (m + mp) * _fft_flops(L) + (2 * q * mp * n * n if xi else 0)
    # per bin and source: the solve (one weight per depth, or two dense real products), and the residual curve
    fl += q * bins * (4 * m * (m + mp) if m > 1 else 2 * mp + 4) + 2 * classes * m * c["alphas"]
    return {"bytes": by, "flops": fl}


def work(case):
    kind = case["kind"]
    if kind == "invert":
        return _work_invert(case)
    if kind == "batch":
        ws = [_work_invert(c) for c in _batch_shapes(case)]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}
    if kind == "forward":
        n, m, mp, q = case["n"], case["planes"], case["depths"], case["sources"]
        el = 8 if case["precision"] == "fp64" else 4
        bins, classes = n * (n // 2 + 1), (n // 2 + 1) * (n // 2 + 2) // 2
        return {"bytes": el * (q * (m + mp) * n * n + classes * m * mp),
                "flops": q * ((m + mp) * _fft_flops(n) + 4 * bins * m * mp)}
    vox = case["batch"] * case["depth"] * case["height"] * case["width"]
    specs = _unet_specs()
    params = sum(ci * co * 27 + co for ci, co, _ in specs) + UNET_WIDTHS[0] + 1
    fl = sum(2 * 27 * ci * co * (vox >> (3 * l)) for ci, co, l in specs)
    if case["what"] == "forward":
        return {"bytes": 4 * (2 * vox + params), "flops": fl}
    first = 2 * 27 * specs[0][1] * vox  # (the first layer has no input gradient)
    return {"bytes": 4 * (2 * vox + 2 * params), "flops": 3 * fl - first}


def exact(case, seed):
    kind = case["kind"]
    if kind == "invert":
        g, A, U, delta = _invert_inputs(case, seed)
        out, _ = _invert_exact(U, g, A, g["alphas"], delta, case["ra"], case["bands"], case["output"])
        return {"out": out, "alpha_idx": None}
    if kind == "batch":
        outs = []
        for k, c in enumerate(_batch_shapes(case)):
            g = _geometry(c)
            A = _kernel_spectra(g)
            U, delta = _data(g, c["noise"], seed * 1000 + k, A)
            outs.append(_invert_exact(U.float(), g, A, g["alphas"], delta)[0])
        return outs
    if kind == "forward":
        g, zeta = _forward_inputs(case, seed)
        return _forward(zeta, _kernel_spectra(g), g)
    x, t = _unet_inputs(case, seed)
    p = torch.tensor(_unet_params(seed), device=_dev()).double().requires_grad_(case["what"] == "gradient")
    s, B = 4.0, case["batch"]
    if case["what"] == "forward":
        with torch.no_grad():
            return torch.stack([_unet_exact(x[b].double(), p, s) / s for b in range(B)])
    loss = 0.0
    for b in range(B):
        ts = s * t[b].double()
        part = (_unet_exact(x[b].double(), p, s) - ts).square().sum() / ts.square().sum() / B
        part.backward()
        loss += float(part.detach())
    return {"grad": p.grad, "loss": torch.tensor([loss], dtype=torch.float64)}
