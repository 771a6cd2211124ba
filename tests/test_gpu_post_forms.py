"""Forms of the FP64 stages at the sizes where they can go wrong: the direct estimator's cells (1e-12
normwise between two forms of the library that add the same terms in another order)."""
import numpy as np
import pytest
import torch

from paper_2309_08601_gb300 import synth
from tests._util import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    from paper_2309_08601_gb300.build import build_native
    build_native()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2309_08601_gb300 import api
    return api


@pytest.mark.parametrize("theta", [[3.0, 3.0, 3.0], [2.0, 2.0, 3.5], [3.5, 2.0, 2.0], [2.0, 3.5, 2.0], [1.5, 2.0, 3.5]])
def test_direct_cells_equal_the_whole_scan(gpu, theta):
    """Many apertures in one call go through the cells, one at a time through the scan of the catalog."""
    cat = synth.make_catalog(5003, 60.0, 3, field="noise", weights="uniform")
    cat.xq[:] -= 200_000  # negative positions
    cat.g1[11] = np.nan  # reaches the apertures that hold the galaxy, no others
    dev = gpu.catalog_to_device(cat)
    off = 200_000 * synth.QUANTUM
    x, y = cat.xq[77] * synth.QUANTUM, cat.yq[77] * synth.QUANTUM
    # outside the field, on a galaxy, a galaxy exactly at the cut-off radius, and a grid
    cen = [[-200.0, 30.0], [x, y], [x + 4.0 * max(theta), y], [59.9 - off, 0.0]]
    cen += [[i - off, j] for i in np.arange(0, 61, 4.0) for j in np.arange(0, 61, 4.0)]
    with gpu.Estimator(n_bins=4, theta_min=1.0, theta_max=8.0, n_max=2) as est:
        many = est.map3_direct(*dev[:5], [theta], cen).cpu().numpy()
        one = np.concatenate([est.map3_direct(*dev[:5], [theta], [c]).cpu().numpy() for c in cen])
    np.testing.assert_array_equal(np.isnan(many), np.isnan(one))
    assert np.isnan(one).any() and not np.isnan(one).all()
    for k in (0, 1):
        ok = ~np.isnan(one[..., k])
        assert rel_err(many[..., k][ok], one[..., k][ok]) < 1e-12
