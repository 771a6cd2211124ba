"""The direct estimator on fields that fill the cell grid unevenly: a distant outlier (the catalog in one
cell), a thin strip (one row of cells), a steep cluster. Many apertures in one call go through the cells, one
at a time through the scan of the catalog: equal to 1e-12 normwise (FP64 sums of the same terms in another
order), repeated runs bitwise. An order within a cell found by n^2 / 4 steps of one thread would take
several seconds here; the calls must end within one."""
import numpy as np
import pytest
import torch

from paper_2309_08601_gb300 import synth
from tests._util import rel_err

pytestmark = pytest.mark.gpu


def _catalog(kind, n=60_011, side=120.0):
    cat = synth.make_catalog(n, side, 3, field="noise", weights="uniform")
    rng = np.random.default_rng(4)
    if kind == "outlier":
        cat.xq[0], cat.yq[0] = 2 ** 31 - 1, -2 ** 31
    elif kind == "strip":
        cat.yq[:] = cat.yq // 4096 + 400_000
    elif kind == "cluster":  # cells from a few to some thousands of galaxies
        r = 20.0 * rng.uniform(size=n) ** 3
        t = rng.uniform(0, 2 * np.pi, n)
        cat.xq[:] = synth.quantise(side / 2 + r * np.cos(t))
        cat.yq[:] = synth.quantise(side / 2 + r * np.sin(t))
    return cat


@pytest.mark.parametrize("theta", [[3.0, 3.0, 3.0], [1.5, 2.0, 3.5]])
@pytest.mark.parametrize("kind", ["outlier", "strip", "cluster"])
def test_uneven_fields(kind, theta):
    from paper_2309_08601_gb300 import api
    from paper_2309_08601_gb300.build import build_native
    build_native()
    cat = _catalog(kind)
    dev = api.catalog_to_device(cat)
    y = float(np.median(cat.yq)) * synth.QUANTUM
    cen = [[x, y + d] for x in np.arange(20.0, 101.0, 10.0) for d in (-7.0, 0.0, 2.0)]
    with api.Estimator(n_bins=4, theta_min=1.0, theta_max=8.0, n_max=2) as est:
        one = np.concatenate([est.map3_direct(*dev[:5], [theta], [c]).cpu().numpy() for c in cen])
        t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t0.record()
        many = est.map3_direct(*dev[:5], [theta], cen)
        t1.record()
        again = est.map3_direct(*dev[:5], [theta], cen)
        many, again = many.cpu().numpy(), again.cpu().numpy()
        assert t0.elapsed_time(t1) < 1000.0
    np.testing.assert_array_equal(many, again)
    assert np.abs(one).max() > 0
    for k in (0, 1):
        assert rel_err(many[..., k], one[..., k]) < 1e-12
