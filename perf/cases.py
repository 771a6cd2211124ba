"""The work a user of this framework has it do, as cases that can be timed.

A measurement is: a catalog's moments (accumulate_moments), their contraction into multipoles
(contract), the FP64 stages after it (edge_correct, to_gamma, to_map3), the whole call (measure),
its gradient (api.map3 and backward), batches of mock catalogs (run_batch), the combined estimator
and the direct estimator. Sizes, binnings and densities are those of the package's workloads
(synth.WORKLOADS) and tests, at areas that keep one pass below two seconds.

The single-precision forms return their multipoles in complex128 arrays that hold the accuracy of
single-precision moments; programs that use these forms keep the results as complex64, as here.
"""
import math

import numpy as np
import torch

from paper_2309_08601_gb300 import api

QUANTUM = 2.0 ** -13  # arcmin per position unit


def listed():
    return [
        # the smallest whole call: 2000 galaxies in FP64, where launches and small kernels count
        dict(name="measure_2k_fp64", kind="measure", n=2000, side=60.0, bins=10, lo=0.5, hi=30.0, n_max=10, z=1,
             precision="fp64", field="noise"),
        # one small mock field in the tensor-core form, called in a loop over many fields
        dict(name="multipoles_3k", kind="multipoles", n=3001, side=60.0, bins=10, lo=0.5, hi=30.0, n_max=10, z=1,
             precision="bf16x3", field="noise"),
        # moments alone of a mid-sized field, every galaxy a centre, read back
        dict(name="moments_20k", kind="moments", n=20_000, side=95.0, bins=20, lo=0.5, hi=60.0, n_max=30, z=1,
             precision="fp32", field="lognormal"),
        # one patch of a wide masked survey: the centres of a rectangle, the members of its halo
        dict(name="moments_patch_masked", kind="moments", n=400_000, side=380.0, bins=30, lo=0.5, hi=240.0, n_max=40,
             z=1, precision="fp32", field="masked", patch=60.0),
        # the benchmark catalog's density and binning, moments and contraction
        dict(name="multipoles_200k", kind="multipoles", n=200_000, side=300.0, bins=20, lo=0.5, hi=120.0, n_max=30, z=1,
             precision="bf16x3", field="lognormal"),
        # tomography: all ordered triplets of five redshift bins
        dict(name="multipoles_tomo5", kind="multipoles", n=40_001, side=100.0, bins=15, lo=0.5, hi=40.0, n_max=20, z=5,
             precision="tf32x3", field="lognormal"),
        # the plain FP64 path at the size used to check the others
        dict(name="multipoles_12k_fp64", kind="multipoles", n=12_000, side=100.0, bins=14, lo=0.5, hi=30.0, n_max=10,
             z=1, precision="fp64", field="lognormal"),
        # combined estimator at the density and binning of its accuracy test
        dict(name="combined_310k", kind="combined", n=310_000, side=190.0, bins=33, lo=0.25, hi=80.0, n_max=30, z=1,
             precision="bf16x3", field="lognormal", fft=False),
        # forward-modelled inference: aperture measures and their gradient per galaxy
        dict(name="gradient_100k", kind="gradient", n=100_000, side=188.0, bins=20, lo=0.5, hi=120.0, n_max=30, z=1,
             precision="bf16x3", field="lognormal"),
        # the FP64 stages after the contraction for 125 redshift triplets
        dict(name="post_tomo5", kind="post", bins=20, lo=0.5, hi=120.0, n_max=30, z=5, n_ap=4),
        # direct estimator on a grid of apertures, the cross-check of the whole route
        dict(name="direct_200k", kind="direct", n=200_000, side=300.0, theta=4.0, theta2=8.0, step=8.0),
        # many small tomographic mock fields through one call
        dict(name="batch_6x3", kind="batch", count=6, n=9000, side=60.0, bins=8, lo=0.5, hi=20.0, n_max=10, z=3,
             precision="fp64", field="lognormal"),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["measure", "multipoles", "multipoles", "moments", "moments", "patch", "combined", "gradient",
                       "post", "direct", "batch"])
    rho = rng.choice([0.55, 1.5, 2.22, 2.78, 4.0, 8.6])  # galaxies per square arcmin
    if kind == "measure":
        n = _log(rng, 1501, 6001)
        side = math.sqrt(n / rho)
        return dict(kind=kind, n=n, side=side, bins=rng.randint(5, 12), lo=0.75, hi=max(6.0, min(30.0, 0.5 * side)),
                    n_max=rng.randint(3, 12), z=rng.choice([1, 1, 2]), precision="fp64",
                    field=rng.choice(["noise", "lognormal"]))
    if kind == "multipoles":
        precision = rng.choice(["bf16x3", "bf16x3", "tf32x3", "fp32", "fp64"])
        n = _log(rng, 701, 12_001 if precision == "fp64" else 120_001)
        side = math.sqrt(n / rho)
        return dict(kind=kind, n=n, side=side, bins=rng.randint(7, 33), lo=0.5, hi=max(6.0, min(120.0, 0.45 * side)),
                    n_max=rng.choice([5, 10, 17, 20, 30] if precision != "fp64" else [5, 8, 10]),
                    z=1 if n > 60_000 else rng.choice([1, 1, 2, 3]), precision=precision,
                    field=rng.choice(["lognormal", "masked"]))
    if kind == "moments":
        n = _log(rng, 501, 60_001)
        side = math.sqrt(n / rho)
        return dict(kind=kind, n=n, side=side, bins=rng.randint(7, 33), lo=0.5, hi=max(6.0, min(120.0, 0.6 * side)),
                    n_max=rng.choice([4, 10, 13, 20, 26, 30, 40, 50]), z=rng.choice([1, 1, 1, 2]), precision="fp32",
                    field=rng.choice(["noise", "lognormal", "masked"]))
    if kind == "patch":
        n = _log(rng, 60_001, 400_001)
        side = math.sqrt(n / max(rho, 1.5))
        return dict(kind="moments", n=n, side=side, bins=rng.randint(15, 33), lo=0.5, hi=min(240.0, 0.4 * side),
                    n_max=rng.choice([10, 20, 30, 40]), z=1, precision="fp32", field=rng.choice(["lognormal", "masked"]),
                    patch=side * rng.uniform(0.08, 0.14))
    if kind == "combined":
        n = _log(rng, 50_001, 310_001)
        return dict(kind=kind, n=n, side=math.sqrt(n / 8.6), bins=rng.randint(20, 33), lo=0.25,
                    hi=min(80.0, 0.42 * math.sqrt(n / 8.6)), n_max=rng.choice([10, 20, 30]), z=1, precision="bf16x3",
                    field="lognormal", fft=rng.random() < 0.5)
    if kind == "gradient":
        n = _log(rng, 801, 100_001)
        side = math.sqrt(n / min(rho, 2.83))
        return dict(kind=kind, n=n, side=side, bins=rng.randint(6, 20), lo=1.5, hi=max(8.0, min(120.0, 0.5 * side)),
                    n_max=rng.choice([5, 10, 20, 30]), z=1, precision="bf16x3", field="lognormal")
    if kind == "post":
        z = rng.choice([1, 2, 3, 5])
        return dict(kind=kind, bins=rng.randint(5, 30 if z < 5 else 20), lo=0.5, hi=rng.choice([30.0, 120.0]),
                    n_max=rng.choice([5, 10, 20, 30] + ([40, 50] if z < 3 else [])), z=z, n_ap=rng.randint(1, 8))
    if kind == "direct":
        n = _log(rng, 2001, 200_001)
        side = max(80.0, math.sqrt(n / rho))
        return dict(kind=kind, n=n, side=side, theta=rng.choice([2.0, 4.0]), theta2=rng.choice([4.0, 8.0]),
                    step=side / rng.uniform(12, 38))
    n = _log(rng, 1501, 12_001)
    return dict(kind="batch", count=rng.randint(2, 6), n=n, side=60.0, bins=rng.randint(5, 10), lo=1.0, hi=20.0,
                n_max=rng.randint(3, 10), z=rng.choice([1, 2, 3]), precision="fp64", field="lognormal")


# ---------------------------------------------------------------------- inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _catalog(case, seed):
    """Device catalog (xq, yq, g1, g2, w, zbin): uniform positions, holes for "masked", lognormal
    Kaiser-Squires shear plus shape noise 0.26 (noise alone for "noise"), weights U(0.5, 1.5)."""
    g, n, side = _gen(seed), case["n"], case["side"]
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    if case.get("field") == "masked":  # holes of 2' to 10' over about 15 % of the area
        nh = max(1, int(0.16 * side * side / (math.pi * 41.0)))
        hx, hy, hr = rand(nh) * side, rand(nh) * side, 2.0 + 8.0 * rand(nh)
        xy = []
        while sum(p.shape[0] for p in xy) < n:
            p = rand(65_536, 2) * side
            d2 = (p[:, :1] - hx) ** 2 + (p[:, 1:] - hy) ** 2
            xy.append(p[(d2 >= hr * hr).all(1)])
        xy = torch.cat(xy)[:n]
    else:
        xy = rand(n, 2) * side
    x, y = xy[:, 0].contiguous(), xy[:, 1].contiguous()
    g1 = 0.26 * torch.randn(n, generator=g, device="cuda")
    g2 = 0.26 * torch.randn(n, generator=g, device="cuda")
    if case.get("field") != "noise":
        m = 2048
        k = torch.fft.fftfreq(m, device="cuda")
        ky, kx = k[:, None], k[None, :]
        k2 = (kx * kx + ky * ky).clamp_min(1e-12)
        amp = k2 ** -0.375
        amp[0, 0] = 0.0
        f = torch.fft.ifft2(torch.fft.fft2(torch.randn(m, m, generator=g, device="cuda")) * amp).real
        f = f / f.std()
        kap = torch.fft.fft2(0.02 * (torch.exp(f - 0.5) - 1.0))
        ks = torch.complex((kx * kx - ky * ky) / k2, 2 * kx * ky / k2)
        ks[0, 0] = 0.0
        gam = torch.fft.ifft2(kap * ks)
        s = gam[(y / side * m).long().clamp(0, m - 1), (x / side * m).long().clamp(0, m - 1)]
        g1, g2 = g1 + s.real, g2 + s.imag
    w = (0.5 + rand(n)).float()
    z = None
    if case.get("z", 1) > 1:
        z = torch.randint(0, case["z"], (n,), generator=g, device="cuda").to(torch.uint8)
    q = lambda v: torch.floor(v / QUANTUM).to(torch.int32).contiguous()  # noqa: E731
    return q(x), q(y), g1.contiguous(), g2.contiguous(), w, z


def _estimator(case):
    return api.Estimator(case["bins"], case["lo"], case["hi"], case["n_max"], n_z=case["z"],
                         precision=case.get("precision", "fp64"), grid_fft=bool(case.get("fft", False)))


def _apertures(case):
    t = [a for a in (2.0, 4.0, 8.0, 16.0) if a < 0.5 * case["hi"]] or [0.25 * case["hi"]]
    return [[a, a, a] for a in t]


def _levels(case):
    """The octave rule of the combined estimator: pixels of 0.25', 0.5', 1' for the bins from 5',
    10', 20' on."""
    edges = case["lo"] * (case["hi"] / case["lo"]) ** (np.arange(case["bins"] + 1) / case["bins"])
    out = []
    for b in range(case["bins"]):
        p = 1.0 if edges[b] >= 20.0 else 0.5 if edges[b] >= 10.0 else 0.25 if edges[b] >= 5.0 else 0.0
        if p and (not out or out[-1][1] != int(round(p / QUANTUM))):
            out.append((b, int(round(p / QUANTUM))))
    return out


def _patch_count(case):
    return int(round(case["n"] * (case["patch"] / case["side"]) ** 2))


def _patch_mask(case, cat):
    """Centres of the patch: the galaxies of a square in the middle of the field."""
    if not case.get("patch"):
        return None
    mid = 0.5 * case["side"] / QUANTUM
    d = torch.maximum((cat[0] - mid).abs(), (cat[1] - mid).abs())
    m = torch.zeros(case["n"], dtype=torch.uint8, device="cuda")
    m[torch.argsort(d, stable=True)[:_patch_count(case)]] = 1
    return m


def _coupling_inputs(case, seed):
    """Multipoles as a contraction leaves them: N and Upsilon summed over 256 centres of a field
    (counts with their scatter for the moments)."""
    g, nb, nm, nz = _gen(seed), case["bins"], case["n_max"], case["z"]
    r = np.geomspace(case["lo"], case["hi"], nb + 1)
    cnt = torch.tensor(2.2 * math.pi * (r[1:] ** 2 - r[:-1] ** 2) + 4.0, device="cuda")
    C = 256

    def noise(*s):
        return torch.complex(torch.randn(*s, generator=g, device="cuda", dtype=torch.float64),
                             torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)) / math.sqrt(2.0)
    W = noise(2 * nm + 1, C, nz, nb) * cnt.sqrt()
    W[0] = cnt * (1.0 + 0.05 * W[0].real / cnt.sqrt())
    G = noise(2, nm + 1, C, nz, nb) * (0.3 * cnt.sqrt())
    v = 0.3 * noise(C, 1, 1)
    norm = torch.einsum("nizb,niyc->nzybc", W, W.conj())
    norm = norm.permute(1, 2, 0, 3, 4)[None].expand(nz, *norm.shape[1:3], 2 * nm + 1, nb, nb)
    norm = norm * (1.0 + 0.1 * torch.arange(nz, device="cuda", dtype=torch.float64))[:, None, None, None, None, None]
    norm = norm.reshape(nz ** 3, 2 * nm + 1, nb, nb).contiguous()
    ups = torch.empty(nz ** 3, 4, nm + 1, nb, nb, dtype=torch.complex128, device="cuda")
    for mu in range(4):
        u = torch.einsum("nizb,niyc->nzybc", G[mu % 2] * v, G[(mu // 2)].conj()).permute(1, 2, 0, 3, 4)
        ups[:, mu] = (u[None].expand(nz, *u.shape) * 1.0).reshape(nz ** 3, nm + 1, nb, nb)
    return ups, norm


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "post":
        s["est"] = _estimator(case)
        s["ups"], s["norm"] = _coupling_inputs(case, seed)
        s["theta"] = [[2.0 * (1 + a), 2.0 * (1 + a), 2.0 * (1 + a)] for a in range(case["n_ap"])]
        return s
    if kind == "direct":
        s["cat"] = _catalog(case, seed)
        s["est"] = api.Estimator(4, 0.5, 8.0, 2)
        s["theta"] = [[case["theta"]] * 3, [case["theta2"]] * 3, [case["theta"], case["theta"], case["theta2"]]]
        s["centres"] = _direct_centres(case)
        return s
    s["est"] = _estimator(case)
    s["theta"] = _apertures(case)
    if kind == "batch":
        s["cats"] = [_catalog(dict(case, n=max(300, int(case["n"] * (1.0 - 0.11 * i)))), 1000 * seed + i)
                     for i in range(case["count"])]
        top = int(case["side"] / QUANTUM)
        s["extent"] = (0, 0, top, top)
        return s
    s["cat"] = _catalog(case, seed)
    s["mask"] = _patch_mask(case, s["cat"])
    if kind == "combined":
        s["levels"] = _levels(case)
    if kind == "gradient":
        s["leaves"] = [t.clone().requires_grad_(True) for t in s["cat"][2:5]]
    return s


def _direct_centres(case):
    m = 4.0 * max(case["theta"], case["theta2"])
    a = np.arange(m, case["side"] - m, case["step"])
    if a.size == 0:
        a = np.array([0.5 * case["side"]])
    X, Y = np.meshgrid(a, a, indexing="ij")
    return np.stack([X.ravel(), Y.ravel()], axis=1)


# ---------------------------------------------------------------------- one pass


def _kept(case, *arrays):
    """The single-precision forms' results as a program keeps them (see the top of the file)."""
    return [a if case.get("precision") == "fp64" else a.to(torch.complex64) for a in arrays]


def run(s):
    case, est = s["case"], s["est"]
    kind = case["kind"]
    if kind == "post":
        gam, _ = est.edge_correct(s["ups"], s["norm"])
        gx, gc = est.to_gamma(gam, 0), est.to_gamma(gam, 1)
        corr, m8 = est.to_map3(gc, s["theta"])
        return [gam, gx, gc, corr, m8]
    if kind == "batch":
        return est.run_batch(s["cats"], s["extent"], s["theta"])
    x, y, g1, g2, w, z = s["cat"]
    if kind == "direct":
        return est.map3_direct(x, y, g1, g2, w, s["theta"], s["centres"])
    if kind == "measure":
        m = est.measure(x, y, g1, g2, w, s["theta"], zbin=z)
        return [m.upsilon, m.norm, m.gamma_n, m.gamma_x, m.gamma_cen, m.corr, m.m8]
    if kind == "gradient":
        a, b, c = s["leaves"]
        m8 = api.map3(est, x, y, a, b, c, s["theta"], zbin=z)
        grads = torch.autograd.grad((1e6 * m8[..., 0]).sum(), (a, b, c))
        return [m8.detach().float(), *grads]  # in the leaves' precision
    if kind == "combined":
        est.accumulate_moments_combined(x, y, g1, g2, w, z, levels=s["levels"])
        return _kept(case, *est.contract())
    est.accumulate_moments(x, y, g1, g2, w, z, centre_mask=s["mask"])
    if kind == "moments":
        return list(est.moments())
    return _kept(case, *est.contract())


# ---------------------------------------------------------------------- what a pass cannot do without


def _pairs(case, centres=None):
    """Expected ordered pairs of a uniform square field between the bins' outer edges."""
    n, L = case["n"], case["side"]

    def inside(r):
        r = min(r, L)
        return math.pi * r * r / L ** 2 - 8.0 / 3.0 * (r / L) ** 3 + 0.5 * (r / L) ** 4
    if centres is not None:  # centres in the middle of the field
        return centres * n * min(1.0, math.pi * case["hi"] ** 2 / L ** 2)
    return float(n) * n * (inside(case["hi"]) - inside(case["lo"]))


def work(case):
    kind = case["kind"]
    if kind == "direct":
        c = _direct_centres(case).shape[0]
        member = case["n"] / case["side"] ** 2 * math.pi * (4.0 * max(case["theta"], case["theta2"])) ** 2
        return {"bytes": 20.0 * case["n"] + 16.0 * c + 48.0 * c, "flops": c * member * 3 * 60.0}
    nb, nm, nz = case["bins"], case["n_max"], case["z"]
    z3, D = nz ** 3, 2 * nm + 1
    ups_b, norm_b = 16.0 * z3 * 4 * (nm + 1) * nb * nb, 16.0 * z3 * D * nb * nb
    gam_b, phi_b = 16.0 * z3 * 4 * D * nb * nb, 16.0 * z3 * 4 * nb * nb * 100
    post = z3 * nb * nb * (8.0 / 3.0 * D ** 3 + 8.0 * 4 * D * D + 2 * 8.0 * 4 * 100 * D)
    if kind == "post":
        return {"bytes": ups_b + norm_b + gam_b + 2 * phi_b, "flops": post}
    if kind == "batch":
        one = work(dict(case, kind="measure"))
        return {"bytes": case["count"] * 21.0 * case["n"], "flops": 0.6 * case["count"] * one["flops"]}
    n = float(case["n"])
    centres = _patch_count(case) if case.get("patch") else None
    nc = centres if centres else n
    el = 16.0 if case.get("precision") == "fp64" else 8.0
    # per pair the separation, the direction and the three sums it enters; per centre and bin the
    # orders; per centre the products of its moments
    flops = 20.0 * _pairs(case, centres) + nc * nz * nb * 6.0 * (4 * nm + 4)
    contraction = nc * nz * nz * nb * nb * 8.0 * (4 * (nm + 1) + D)
    if kind == "moments":
        return {"bytes": 21.0 * n + el * nc * nz * nb * (4 * nm + 4), "flops": flops}
    small = 1.0 if el == 16.0 else 0.5
    if kind == "combined":  # the pixels' pairs are far fewer than the galaxies'
        flops = 20.0 * 0.05 * _pairs(case) + n * nb * 6.0 * (4 * nm + 4)
    if kind in ("multipoles", "combined"):
        return {"bytes": 21.0 * n + small * (ups_b + norm_b), "flops": flops + contraction}
    if kind == "gradient":
        return {"bytes": 32.0 * n, "flops": 2.0 * flops + 3.0 * contraction + 2.0 * post}
    return {"bytes": 21.0 * n + ups_b + norm_b + gam_b + 2 * phi_b, "flops": flops + contraction + post}


# ---------------------------------------------------------------------- the same in 64 bits

CD = torch.complex128


def _edges(case):
    b = np.arange(case["bins"] + 1)
    e = np.array([case["lo"] * math.pow(case["hi"] / case["lo"], float(i) / case["bins"]) for i in b])
    return e, torch.tensor(np.ceil((e / QUANTUM) ** 2).astype(np.int64), device="cuda")


def _chunks(case, cat, idx):
    """For chunks of centres: (their indexes, the mask of every (bin and z-bin) [c][z nb][n] in
    FP64, z = e^{i phi} [c][n])."""
    x, y = cat[0].long(), cat[1].long()
    nz, nb, n = case["z"], case["bins"], x.numel()
    _, e2 = _edges(case)
    zb = cat[5].long() if nz > 1 else torch.zeros_like(x)
    step = max(1, int(2.5e8 // (n * (nz * nb + 30))))
    for i0 in range(0, idx.numel(), step):
        c = idx[i0:i0 + step]
        dx, dy = x[None] - x[c, None], y[None] - y[c, None]
        r2 = dx * dx + dy * dy
        b = torch.bucketize(r2, e2, right=True) - 1
        ok = (b >= 0) & (b < nb)
        key = torch.where(ok, zb[None] * nb + b, nz * nb)
        mask = torch.zeros(c.numel(), nz * nb + 1, n, dtype=torch.float64, device="cuda")
        mask.scatter_(1, key[:, None], 1.0)
        r = r2.double().sqrt().clamp_min(1.0)
        yield c, mask[:, :-1], torch.complex(dx / r, dy / r)


def _powers(z, m):
    """(m, z^m) for m = 0..m: by squares and products of one lower power each."""
    p = torch.ones_like(z)
    yield 0, p
    for i in range(1, m + 1):
        p = p * z
        if i % 8 == 0:  # back onto the unit circle
            p = p / p.abs().clamp_min(1e-300)
        yield i, p


def _exact_moments(case, cat, idx):
    """G [c][z][b][2 n_max + 3] and W [c][z][b][2 n_max + 1] in complex128."""
    nz, nb, nm = case["z"], case["bins"], case["n_max"]
    g1, g2, w = (t.double() for t in cat[2:5])
    G = torch.empty(idx.numel(), nz * nb, 2 * nm + 3, dtype=CD, device="cuda")
    W = torch.empty(idx.numel(), nz * nb, 2 * nm + 1, dtype=CD, device="cuda")
    at = 0
    for c, mask, z in _chunks(case, cat, idx):
        s = slice(at, at + c.numel())
        for m, p in _powers(z, max(2 * nm, nm + 3)):
            cols = [w * p.real, w * p.imag]
            if m <= nm + 3:
                cols += [w * g1 * p.real, w * g1 * p.imag, w * g2 * p.real, w * g2 * p.imag]
            v = torch.bmm(mask, torch.stack(cols, 2))
            if m <= 2 * nm:
                W[s, :, m] = torch.complex(v[..., 0], v[..., 1])
            if m <= nm + 3:
                A, B = torch.complex(v[..., 2], v[..., 3]), torch.complex(v[..., 4], v[..., 5])
                if m <= nm - 1:
                    G[s, :, m + nm + 3] = A + 1j * B
                if m > 0:
                    G[s, :, nm + 3 - m] = A.conj() + 1j * B.conj()
        at += c.numel()
    return G.view(-1, nz, nb, 2 * nm + 3), W.view(-1, nz, nb, 2 * nm + 1)


def _exact_contract(case, cat, G, W):
    nz, nb, nm, o = case["z"], case["bins"], case["n_max"], case["n_max"] + 3
    v = torch.complex(*(cat[4].double() * t.double() for t in cat[2:4]))
    w = cat[4].double()
    zb = cat[5].long() if nz > 1 else torch.zeros(w.numel(), dtype=torch.int64, device="cuda")
    ups = torch.zeros(nz ** 3, 4, nm + 1, nb, nb, dtype=CD, device="cuda")
    norm = torch.zeros(nz ** 3, 2 * nm + 1, nb, nb, dtype=CD, device="cuda")

    def dot(c, X, Y):
        return (c[:, None] * X).transpose(0, 1) @ Y
    for z1 in range(nz):
        sel = zb == z1
        g, ww, c, cw = G[sel], W[sel], v[sel], w[sel].to(CD)
        for z2 in range(nz):
            for z3 in range(nz):
                t = (z1 * nz + z2) * nz + z3
                for n in range(nm + 1):
                    a, b = (lambda m: g[:, z2, :, m + o]), (lambda m: g[:, z3, :, m + o])
                    ups[t, 0, n] = -dot(c, a(n - 3), b(-n - 3))
                    ups[t, 1, n] = -dot(c.conj(), a(n - 1), b(-n - 1))
                    ups[t, 2, n] = -dot(c, a(-n - 1).conj(), b(-n - 3))
                    ups[t, 3, n] = -dot(c, a(n - 3), b(n - 1).conj())
                for n in range(2 * nm + 1):
                    norm[t, n] = dot(cw, ww[:, z2, :, n], ww[:, z3, :, n].conj())
    return ups, norm


def _exact_edge(case, ups, norm):
    """Gamma_n of sum_n N_{l-n} Gamma_n = Upsilon_l, the negative orders by the symmetries."""
    nz, nb, nm = case["z"], case["bins"], case["n_max"]
    sw = torch.arange(nz ** 3, device="cuda").view(nz, nz, nz).transpose(1, 2).reshape(-1)
    Un = ups[sw][:, [0, 1, 3, 2]].transpose(-1, -2)
    U = torch.cat([Un[:, :, 1:].flip(2), ups], 2)  # [t][mu][l][b1][b2]
    Nn = norm[sw].transpose(-1, -2)
    N = torch.cat([Nn[:, 1:].flip(1), norm], 1)  # m = -2 n_max .. 2 n_max
    l = torch.arange(2 * nm + 1, device="cuda")
    out = torch.empty(nz ** 3, 4, 2 * nm + 1, nb, nb, dtype=CD, device="cuda")
    for t in range(nz ** 3):
        A = N[t][(l[:, None] - l[None]) + 2 * nm].permute(2, 3, 0, 1)
        out[t] = torch.linalg.solve(A, U[t].permute(2, 3, 1, 0)).permute(3, 2, 0, 1)
    return out


def _nodes(case):
    e, _ = _edges(case)
    t = torch.tensor(0.5 * (e[1:] + e[:-1]), device="cuda")
    return t, torch.tensor(np.diff(e), device="cuda")


def _exact_gamma(case, gam):
    nm, nphi = case["n_max"], 100
    phi = (torch.arange(nphi, device="cuda", dtype=torch.float64) + 0.5) * (2 * math.pi / nphi)
    n = torch.arange(-nm, nm + 1, device="cuda", dtype=torch.float64)
    ph = n[:, None] * phi[None]
    gx = torch.einsum("tmnbc,nk->tmbck", gam, torch.complex(ph.cos(), ph.sin()))
    t, _ = _nodes(case)
    e = torch.complex(phi.cos(), phi.sin())
    t1, t2 = t[:, None, None], t[None, :, None]
    unit = lambda q: q.conj() / q  # noqa: E731
    r1, r2, r3 = unit(t1 + t2 * e), unit(t2 * e - 2 * t1), unit(t1 - 2 * t2 * e)
    f = torch.stack([r1 * r2 * r3 * e ** 3, r2 * r3 / r1 * e, r1 * r3 / r2 * e ** 3, r1 * r2 / r3 * e.conj()])
    return gx, gx * f


def _exact_map3(case, gc, theta):
    """Aperture correlators and the eight real measures by the midpoint rule."""
    nphi = 100
    phi = (torch.arange(nphi, device="cuda", dtype=torch.float64) + 0.5) * (2 * math.pi / nphi)
    e = torch.complex(phi.cos(), phi.sin())
    t, dt = _nodes(case)
    t1, t2 = t[:, None, None].to(CD), t[None, :, None] * e
    q = [-(t1 + t2) / 3, (2 * t1 - t2) / 3, (2 * t2 - t1) / 3]
    wgt = dt[:, None, None] * dt[None, :, None] * (2 * math.pi / nphi)
    corr = torch.empty(gc.shape[0], len(theta), 4, dtype=CD, device="cuda")
    for a, th in enumerate(theta):
        s = [float(v) ** 2 for v in th]
        T4 = (s[0] * s[1] + s[0] * s[2] + s[1] * s[2]) / 3
        T2 = math.sqrt(T4)
        q2 = [(v.abs() ** 2) for v in q]
        f, g, Z = [], [], 0.0
        for i in range(3):
            j, k = (i + 1) % 3, (i + 2) % 3
            r = q[i].conj() * (q[j] - q[k]) / q2[i]
            f.append((s[j] + s[k]) / (2 * T2) + r * (s[j] - s[k]) / (6 * T2))
            g.append(s[j] * s[k] / T4 + r * s[i] * (s[k] - s[j]) / (3 * T4))
            Z = Z + (-s[i] + 2 * s[j] + 2 * s[k]) * q2[i]
        pre = s[0] * s[1] * s[2] / (T2 * T4) / (2 * math.pi * T4) * t[:, None, None] * t[None, :, None] * torch.exp(
            -Z / (6 * T4))
        aq = q2[0] * q2[1] * q2[2]
        F = [pre * aq / (24 * T2 * T4) * (f[0] * f[1] * f[2]).conj() ** 2]
        for mu in (1, 2, 3):
            i, j, k = (mu + 1) % 3, (mu + 2) % 3, mu % 3  # the conjugate's vertex is j
            ff, qq = (f[k] * f[i]).conj(), q[k] * q[i] * q[j].conj() ** 2
            F.append(pre * (aq / (24 * T2 * T4) * ff ** 2 * f[j] ** 2 - qq / (9 * T4) * ff * f[j] * g[j].conj()
                            + (qq ** 2 / (aq * T2) * g[j].conj() ** 2
                               + 2 * s[k] * s[i] / (T4 * T2) * qq / q2[j] * ff) / 27))
        for mu in range(4):
            corr[:, a, mu] = (gc[:, mu] * F[mu] * wgt).sum((1, 2, 3))
    c0, c1, c2, c3 = corr.unbind(-1)
    r0, r1, r2, r3, i0, i1, i2, i3 = (*(c.real for c in (c0, c1, c2, c3)), *(c.imag for c in (c0, c1, c2, c3)))
    m8 = torch.stack([r3 + r2 + r1 + r0, i3 + i2 - i1 + i0, i3 - i2 + i1 + i0, -i3 + i2 + i1 + i0,
                      r3 + r2 - r1 - r0, r3 - r2 + r1 - r0, -r3 + r2 + r1 - r0, i3 + i2 + i1 - i0], -1) / 4
    return corr, m8


def _exact_gradient(case, cat, theta):
    """m8 and dL/d(g1, g2, w): autograd from the moments on, the moments' own (linear) adjoint by
    sums over pairs."""
    nz, nb, nm = case["z"], case["bins"], case["n_max"]
    idx = torch.arange(cat[0].numel(), device="cuda")
    G, W = _exact_moments(case, cat, idx)
    G.requires_grad_(True), W.requires_grad_(True)
    p = [t.double().requires_grad_(True) for t in cat[2:5]]
    ups, norm = _exact_contract(case, (*cat[:2], *p, cat[5]), G, W)
    gam = _exact_edge(case, ups, norm)
    m8 = _exact_map3(case, _exact_gamma(case, gam)[1], theta)[1]
    gG, gW, d1, d2, dw = torch.autograd.grad((1e6 * m8[..., 0]).sum(), (G, W, *p))
    g1, g2, w = (t.detach() for t in p)
    gG, gW = gG.reshape(len(idx), nz * nb, -1), gW.reshape(len(idx), nz * nb, -1)
    gv = torch.zeros(w.numel(), dtype=CD, device="cuda")
    gw = torch.zeros_like(w)
    at = 0
    for c, mask, z in _chunks(case, cat, idx):
        s, mt = slice(at, at + c.numel()), mask.to(CD).transpose(1, 2)
        for m, u in _powers(z, max(2 * nm, nm + 3)):
            if m <= 2 * nm:
                gw += ((mt @ gW[s, :, m, None])[..., 0] * u.conj()).real.sum(0)
            if m <= nm - 1:
                gv += ((mt @ gG[s, :, m + nm + 3, None])[..., 0] * u.conj()).sum(0)
            if 0 < m <= nm + 3:
                gv += ((mt @ gG[s, :, nm + 3 - m, None])[..., 0] * u).sum(0)
        at += c.numel()
    return [m8.detach(), d1 + w * gv.real, d2 + w * gv.imag, dw + gw + g1 * gv.real + g2 * gv.imag]


def _exact_direct(case, cat, theta, centres):
    x, y = cat[0].double() * QUANTUM, cat[1].double() * QUANTUM
    g1, g2, w = (t.double() for t in cat[2:5])
    cen = torch.tensor(centres, device="cuda")
    out = torch.empty(len(centres), len(theta), 2, dtype=torch.float64, device="cuda")
    step = max(1, int(4e7 // x.numel()))
    for i in range(0, len(centres), step):
        dx, dy = x[None] - cen[i:i + step, :1], y[None] - cen[i:i + step, 1:]
        r2 = dx * dx + dy * dy
        gt = -(g1 * (dx * dx - dy * dy) + 2 * g2 * dx * dy) / r2.clamp_min(1e-300)
        for a, th in enumerate(theta):
            keep = (r2 > 0) & (r2.sqrt() <= 4.0 * max(th))
            b = [torch.where(keep, w * r2 / (4 * math.pi * t ** 4) * torch.exp(-r2 / (2 * t * t)), 0.0) for t in th]
            for k, f in enumerate(([v * gt for v in b], b)):
                s = lambda *v: math.prod(v[1:], start=v[0]).sum(1)  # noqa: E731
                p, q, r = f
                out[i:i + step, a, k] = (s(p) * s(q) * s(r) - s(p, q) * s(r) - s(p, r) * s(q) - s(q, r) * s(p)
                                         + 2 * s(p, q, r))
    return out


def _exact_cost(case):
    """Seconds the exact moments take, roughly (FP64 products with the bins' masks)."""
    nz, nb, nm = case["z"], case["bins"], case["n_max"]
    nc = _patch_count(case) if case.get("patch") else case["n"]
    return nc * case["n"] * ((6 * nm + 26) * (2.0 * nz * nb + 40) + 30 * nz * nb) / 0.5e12


def exact(case, seed):
    kind = case["kind"]
    if kind == "combined":
        return None
    if kind == "direct":
        if case["n"] * float(_direct_centres(case).shape[0]) > 6e8:
            return None
        s = prepare(case, seed)
        return _exact_direct(case, s["cat"], s["theta"], s["centres"])
    if kind == "post":
        s = prepare(case, seed)
        gam = _exact_edge(case, s["ups"], s["norm"])
        gx, gc = _exact_gamma(case, gam)
        return [gam, gx, gc, *_exact_map3(case, gc, s["theta"])]
    if _exact_cost(case) * case.get("count", 1) * (3.0 if kind == "gradient" else 1.0) > 16.0:
        return None
    s = prepare(case, seed)
    if kind == "batch":
        return torch.stack([_exact_chain(case, c, s["theta"])[-1] for c in s["cats"]])
    if kind == "gradient":
        return _exact_gradient(case, s["cat"], s["theta"]) if case["n"] <= 6000 else None
    if kind == "measure":
        return _exact_chain(case, s["cat"], s["theta"])
    n = s["cat"][0].numel()
    idx = torch.arange(n, device="cuda") if s["mask"] is None else s["mask"].nonzero()[:, 0]
    G, W = _exact_moments(case, s["cat"], idx)
    if kind == "moments":
        return [G, W]
    return list(_exact_contract(case, s["cat"], G, W))


def _exact_chain(case, cat, theta):
    G, W = _exact_moments(case, cat, torch.arange(cat[0].numel(), device="cuda"))
    ups, norm = _exact_contract(case, cat, G, W)
    gam = _exact_edge(case, ups, norm)
    gx, gc = _exact_gamma(case, gam)
    return [ups, norm, gam, gx, gc, *_exact_map3(case, gc, theta)]
