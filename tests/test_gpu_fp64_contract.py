"""The FP64 contraction (csrc/contract.cu), which forms half of the normalisation's Hermitian blocks,
against the oracle's contraction of its own moments: odd and even bin counts, more outputs than
threads, equal and unequal redshift bins, added to what the buffers hold. Tolerance, normwise: sums of
at most 300 centres' products of sums of at most 300 neighbours, each off by less than 600 2^-53: 1e-12.
"""
import numpy as np
import pytest
import torch

from paper_2309_08601_gb300 import synth
from tests._util import rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bins,n_max,n_z", [(1, 0, 1), (2, 3, 2), (7, 4, 3), (16, 2, 1), (17, 3, 2), (33, 2, 1)])
def test_fp64_contraction(orc, n_bins, n_max, n_z):
    from paper_2309_08601_gb300 import api
    from paper_2309_08601_gb300.build import build_native
    build_native()
    cat = synth.make_catalog(300, 12.0, 5 + n_bins, field="noise", weights="uniform")
    if n_z > 1:
        cat.zbin = np.random.default_rng(n_bins).integers(0, n_z, cat.n).astype(np.uint8)
    s = orc.Setup(n_bins=n_bins, theta_min=0.5, theta_max=8.0, n_max=n_max, n_z=n_z)
    ups, norm = orc.contract(s, cat, *orc.moments(s, cat))
    with api.Estimator(n_bins, 0.5, 8.0, n_max, n_z=n_z, precision="fp64") as est:
        est.accumulate_moments(*api.catalog_to_device(cat))
        u, m = est.contract()
        assert rel_err(u.cpu().numpy(), ups) < 1e-12
        assert rel_err(m.cpu().numpy(), norm) < 1e-12
        est.contract(u, m)
        assert rel_err(m.cpu().numpy(), 2 * norm) < 1e-12
        assert torch.isfinite(torch.view_as_real(m)).all()
