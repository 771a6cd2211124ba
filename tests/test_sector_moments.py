"""The moments of wide radial bins by angular sectors (csrc/moments_far.cu, csrc/sector.cuh).

On the CPU: every galaxy within an annulus is listed exactly once over the sectors, for groups,
cells and annuli of many shapes. On the GPU: moments and pair counts against the FP64 path, which
takes every pair through the direct form. Tolerance, normwise per array: a direction in FP32 is off
by about 1.5 2^-24, an order m <= 100 by m times that (9e-6 if all pairs erred alike), the dropped
Chebyshev terms add 3e-8: 1e-5. That holds for the bins of the sector form, here those with 2000
expected neighbours; the bins nearer to the centre take the direct form, whose order recurrence
alone may be 1.4e-5 off, and are held to the FP32 path's 1e-4.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2309_08601_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def runs(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path_factory.mktemp("sector") / "sector_runs")
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I" + os.path.join(ROOT, "include"), "-o",
                    exe, os.path.join(ROOT, "tests", "c", "sector_runs.cu")], check=True)
    return exe


@pytest.mark.parametrize("args", [
    "1 20000 5000 140 140 64 3 4 150000 200000 0", "2 20000 5000 140 140 64 3 4 400000 900000 1",
    "3 5000 20000 70 71 64 4 5 500000 600000 0", "4 9000 137 95 95 32 1 1 3000 4000 0",
    "5 30000 100000 160 160 64 3 4 3e6 9e6 1", "6 3000 1 60 61 64 3 4 40 50 0", "7 4000 3 200 7 32 1 2 100 101 0",
    "8 4000 7919 1 300 64 2 1 150000 700000 0"])
def test_every_galaxy_is_in_one_sector(runs, args):
    r = subprocess.run([runs] + args.split(), capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 0


CASES = {
    "n30": dict(n=20011, side=60.0, hi=40.0, bins=16, n_max=30),
    "n10": dict(n=20011, side=60.0, hi=40.0, bins=11, n_max=10),
    "n3": dict(n=6001, side=40.0, hi=30.0, bins=9, n_max=3),
    "n0": dict(n=6001, side=40.0, hi=30.0, bins=9, n_max=0),
    "n50": dict(n=20011, side=50.0, hi=45.0, bins=9, n_max=50),
    "tomography": dict(n=30011, side=60.0, hi=45.0, bins=9, n_max=17, n_z=2),
    "holes": dict(n=20011, side=80.0, hi=60.0, bins=14, n_max=26, holes=True),
    "patch": dict(n=60011, side=120.0, hi=50.0, bins=14, n_max=30, centres="patch"),
    "sparse centres": dict(n=20011, side=60.0, hi=40.0, bins=14, n_max=20, centres="sparse"),
    "no centre": dict(n=6001, side=40.0, hi=30.0, bins=9, n_max=10, centres="none"),
    "clusters": dict(n=20011, side=60.0, hi=40.0, bins=14, n_max=30, clusters=True),
    "strip": dict(n=20011, side=150.0, hi=70.0, bins=12, n_max=30, flat=True),
    "coarse cells": dict(n=20011, side=60.0, hi=40.0, bins=12, n_max=30, cell_occupancy=9),
    "extent": dict(n=20011, side=60.0, hi=40.0, bins=12, n_max=30, extent=True),
    "wide": dict(n=250_007, side=200.0, hi=140.0, bins=8, lo=20.0, n_max=30, centres="patch"),
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", CASES)
def test_sector_moments_match_the_direct_form(name):
    import torch
    from paper_2309_08601_gb300 import api
    from paper_2309_08601_gb300.build import build_native
    build_native()
    c = CASES[name]
    rng = np.random.default_rng(sum(map(ord, name)))
    cat = synth.make_catalog(c["n"], c["side"], 5, field="noise", weights="uniform", holes=c.get("holes", False))
    if c.get("clusters"):  # half of the galaxies in twelve dense clumps
        k = cat.n // 2
        at = rng.uniform(5, c["side"] - 5, (12, 2))[rng.integers(0, 12, k)] + rng.normal(0, 0.7, (k, 2))
        cat.xq[:k], cat.yq[:k] = synth.quantise(at[:, 0]), synth.quantise(at[:, 1])
    if c.get("flat"):
        cat.yq[:] = (cat.yq * 0.05).astype(np.int32)
    nz = c.get("n_z", 1)
    if nz > 1:
        cat.zbin = rng.integers(0, nz, cat.n).astype(np.uint8)
    mask = np.ones(cat.n, np.uint8)
    if c.get("centres") == "patch":
        q = c["side"] / synth.QUANTUM
        mask = ((np.abs(cat.xq - 0.4 * q) < 0.06 * q) & (np.abs(cat.yq - 0.5 * q) < 0.05 * q)).astype(np.uint8)
    elif c.get("centres") == "sparse":
        mask = (rng.uniform(size=cat.n) < 0.02).astype(np.uint8)
    elif c.get("centres") == "none":
        mask[:] = 0
    dev = api.catalog_to_device(cat)
    dm = torch.as_tensor(mask, device="cuda") if "centres" in c else None
    out = {}
    for precision in ("fp32", "fp64"):
        with api.Estimator(c["bins"], c.get("lo", 0.5), c["hi"], c["n_max"], n_z=nz, precision=precision,
                           cell_occupancy=c.get("cell_occupancy", 0)) as est:
            if c.get("extent"):
                est.set_extent((-5000, -7000, int(c["side"] / synth.QUANTUM) + 9000, int(c["side"] / synth.QUANTUM)))
            est.accumulate_moments(*dev, centre_mask=dm)
            counts = est.counts()
            out[precision] = (counts, *[t.cpu().numpy() for t in est.moments()])
            if precision == "fp32":  # the same sums in the same order
                est.accumulate_moments(*dev, centre_mask=dm)
                for a, b in zip(out[precision][1:], est.moments()):
                    np.testing.assert_array_equal(a, b.cpu().numpy())
    assert out["fp32"][0] == out["fp64"][0]  # the same pairs
    assert out["fp64"][0][0] == int(mask.sum())
    lo = c.get("lo", 0.5)
    edges = lo * (c["hi"] / lo) ** (np.arange(c["bins"] + 1) / c["bins"])
    rho = cat.n / nz * synth.QUANTUM ** -2 / (np.ptp(cat.xq) + 1.0) / (np.ptp(cat.yq) + 1.0)
    for a, b in zip(out["fp32"][1:], out["fp64"][1:]):
        for i in range(a.shape[2]):  # bin by bin
            err = np.abs(a[:, :, i] - b[:, :, i]).max(initial=0.0)
            wide = np.pi * rho * (edges[i + 1] ** 2 - edges[i] ** 2) > 2000
            assert err <= (1e-5 if wide else 1e-4) * np.abs(b[:, :, i]).max(initial=0.0), (i, wide, err)


@pytest.mark.gpu
def test_non_finite_shears_stay_in_their_bins():
    """A NaN shear reaches the moments of the (centre, bin)s that contain its galaxy and no others."""
    import torch
    from paper_2309_08601_gb300 import api
    from paper_2309_08601_gb300.build import build_native
    build_native()
    cat = synth.make_catalog(20011, 60.0, 5, field="noise", weights="uniform")
    cat.g1[7] = np.nan
    dev = api.catalog_to_device(cat)
    bad = []
    for precision in ("fp32", "fp64"):
        with api.Estimator(12, 0.5, 40.0, 30, precision=precision) as est:
            est.accumulate_moments(*dev)
            G, W = est.moments()
            assert bool(torch.isfinite(torch.view_as_real(W)).all())
            bad.append((~torch.isfinite(torch.view_as_real(G)).all(-1)).any(-1).cpu().numpy())
    assert bad[0].any()
    np.testing.assert_array_equal(bad[0], bad[1])
