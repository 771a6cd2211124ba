"""The moments of narrow bins (csrc/moments_near.cu) against the FP64 oracle at the edges of the orders
that its lanes hold (16 a half-warp and step), with none, one and odd numbers of members, over more than
one batch of 32 and more than one z-bin. Tolerance, normwise per array: FP64 1e-12; FP32 a direction is
off by about 1.5 2^-24 and a power m by m times that, and its products by another 2 ulp: (1.5 m + 2)
2^-24 at the highest order m, plus the sum's 2^-24 a step over at most 100 members.
"""
import numpy as np
import pytest

from paper_2309_08601_gb300 import synth
from tests._util import rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n_max,n_z", [(0, 1), (3, 1), (7, 2), (8, 1), (12, 1), (13, 1), (15, 3), (16, 1), (23, 1), (24, 1),
                                       (30, 2), (31, 1), (32, 1), (47, 1), (48, 1), (50, 2)])
def test_narrow_bins(orc, n_max, n_z, precision):
    from paper_2309_08601_gb300 import api
    from paper_2309_08601_gb300.build import build_native
    build_native()
    cat = synth.make_catalog(1500, 12.0, 5 + n_max, field="noise", weights="uniform")
    if n_z > 1:
        cat.zbin = np.random.default_rng(n_max).integers(0, n_z, cat.n).astype(np.uint8)
    s = orc.Setup(n_bins=6, theta_min=0.02, theta_max=1.5, n_max=n_max, n_z=n_z)
    G, W = orc.moments(s, cat)
    with api.Estimator(6, 0.02, 1.5, n_max, n_z=n_z, precision=precision) as est:
        est.accumulate_moments(*api.catalog_to_device(cat))
        got = [t.cpu().numpy() for t in est.moments()]
    top = max(2 * n_max, n_max + 3)
    tol = 1e-12 if precision == "fp64" else (1.5 * top + 2 + 100) * 2.0 ** -24
    assert rel_err(got[0], G) < tol and rel_err(got[1], W) < tol
