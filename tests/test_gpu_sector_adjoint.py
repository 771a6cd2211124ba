"""The adjoint of the sector form (far_moments_kernel<PL, true>, csrc/moments_far.cu) galaxy by galaxy: the
gradients of the FP32 form, whose wide bins go through it, against the FP64 form's, where the pair kernel takes
every bin. Random dL/dUpsilon and dL/dN. 1e-4 normwise per array, the differentiation form's tolerance in FP32.
Each case states how many of the four sector variants its plan must reach, so that it cannot miss the kernel."""
import numpy as np
import pytest
import torch

from paper_2309_08601_gb300 import synth
from tests._util import rel_err

pytestmark = pytest.mark.gpu

CASES = {
    "n30": dict(n=20011, side=60.0, lo=0.5, hi=40.0, bins=16, n_max=30, variants=3),
    "n10": dict(n=20011, side=60.0, lo=0.5, hi=40.0, bins=11, n_max=10, variants=1),
    "n50": dict(n=40011, side=50.0, lo=2.0, hi=45.0, bins=9, n_max=50, variants=2),
    "tomography": dict(n=30011, side=60.0, lo=0.5, hi=45.0, bins=9, n_max=17, n_z=2, variants=3),
    "strip": dict(n=20011, side=150.0, lo=0.5, hi=70.0, bins=12, n_max=30, flat=True, variants=4),
    "coarse cells": dict(n=20011, side=60.0, lo=0.5, hi=40.0, bins=12, n_max=30, cell_occupancy=9, variants=2),
    "patch": dict(n=60011, side=120.0, lo=1.0, hi=50.0, bins=14, n_max=30, centres=True, variants=4),
    "holes": dict(n=20011, side=60.0, lo=0.5, hi=40.0, bins=16, n_max=30, holes=True, variants=3),
}


@pytest.mark.parametrize("name", CASES)
def test_gradient_of_every_galaxy(name):
    from paper_2309_08601_gb300 import api
    from paper_2309_08601_gb300.build import build_native
    build_native()
    c = CASES[name]
    rng = np.random.default_rng(sum(map(ord, name)))
    cat = synth.make_catalog(c["n"], c["side"], 5, field="noise", weights="uniform", holes=c.get("holes", False))
    if c.get("flat"):
        cat.yq[:] = (cat.yq * 0.05).astype(np.int32)
    nz = c.get("n_z", 1)
    if nz > 1:
        cat.zbin = rng.integers(0, nz, cat.n).astype(np.uint8)
    mask = None
    if c.get("centres"):
        q = c["side"] / synth.QUANTUM
        inside = (np.abs(cat.xq - 0.4 * q) < 0.06 * q) & (np.abs(cat.yq - 0.5 * q) < 0.05 * q)
        mask = torch.as_tensor(inside.astype(np.uint8)).cuda()
    dev = api.catalog_to_device(cat)
    grad = {}
    for precision in ("fp64", "fp32"):
        with api.Estimator(c["bins"], c["lo"], c["hi"], c["n_max"], n_z=nz, precision=precision,
                           cell_occupancy=c.get("cell_occupancy", 0)) as est:
            est.accumulate_moments(*dev, centre_mask=mask)
            if precision == "fp64":
                gu, gn = (torch.complex(*[torch.as_tensor(rng.normal(size=tuple(t.shape))) for _ in range(2)]).cuda()
                          for t in est.new_multipoles())
            est.stage_times()
            grad[precision] = [t.cpu().numpy() for t in est.moments_adjoint(gu, gn, *dev[2:5])]
            launches = est.stage_times()["moments"][1]
            if precision == "fp32":
                assert launches - 4 >= c["variants"]
    for a, b in zip(grad["fp32"], grad["fp64"]):
        err = rel_err(a, b)
        print(name, err)
        assert err < 1e-4
