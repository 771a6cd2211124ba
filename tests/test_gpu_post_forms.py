"""The FP64 stages' forms: angular nodes folded by symmetry (to_gamma), filters tabulated per radii
triple (to_map3) and the direct estimator's cells, at the sizes where they can go wrong. FP64
throughout: 1e-10 normwise, the tolerance of the FP64 path (1e-12 between two forms of the library
that add the same terms in another order)."""
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


def _gamma_n(nz, nb, n_max, seed):
    rng = np.random.default_rng(seed)
    shape = (nz ** 3, 4, 2 * n_max + 1, nb, nb)
    return rng.normal(size=shape) + 1j * rng.normal(size=shape)


@pytest.mark.parametrize("n_phi", [1, 2, 3, 6, 7, 10, 33, 100, 514, 1030])
@pytest.mark.parametrize("nz, nb, n_max", [(1, 3, 0), (1, 7, 5), (2, 3, 4), (3, 2, 1)])
def test_to_gamma_folds_every_node(gpu, orc, nz, nb, n_max, n_phi):
    setup = dict(n_bins=nb, theta_min=0.7, theta_max=9.0, n_max=n_max, n_phi=n_phi, n_z=nz)
    g = _gamma_n(nz, nb, n_max, n_phi)
    g[0, 1, :, 0, nb - 1] = np.nan  # a singular system stays in its own cell
    with gpu.Estimator(**setup, precision="fp64") as est:
        for proj in (0, 1, 2):
            want = orc.to_gamma(orc.Setup(**setup), g, proj)
            got = est.to_gamma(torch.as_tensor(g, device="cuda"), proj).cpu().numpy()
            if proj == 1 and n_phi % 2:
                # node phi = pi, equal radii: the third vertex on the first, where the centroid factor is
                # 0 / 0 (the GPU's cos pi is -1 exactly, the oracle's sin pi is not 0)
                i = np.arange(nb)
                want[:, :, i, i, n_phi // 2] = np.nan
            np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
            ok = ~np.isnan(want)
            assert rel_err(got[ok], want[ok]) < 1e-10, proj


@pytest.mark.parametrize("n_phi", [36, 37])
@pytest.mark.parametrize("nz, n_ap", [(1, 1), (1, 4), (1, 5), (2, 3), (2, 9)])
def test_to_map3_by_tabulated_filters(gpu, orc, nz, n_ap, n_phi):
    setup = dict(n_bins=5, theta_min=0.5, theta_max=12.0, n_max=3, n_phi=n_phi, n_z=nz)
    rng = np.random.default_rng(n_ap)
    shape = (nz ** 3, 4, 5, 5, n_phi)
    gc = rng.normal(size=shape) + 1j * rng.normal(size=shape)
    th = rng.uniform(1.0, 4.0, (n_ap, 3))
    corr, m8 = orc.to_map3(orc.Setup(**setup), gc, th)
    with gpu.Estimator(**setup, precision="fp64") as est:
        gcorr, gm8 = est.to_map3(torch.as_tensor(gc, device="cuda"), th)
    if n_phi % 2:  # the node phi = pi with equal radii is 0 / 0 in the filter on the GPU
        assert bool(torch.isnan(gm8).all()) and bool(torch.isnan(torch.view_as_real(gcorr)).all())
        return
    assert rel_err(gcorr.cpu().numpy(), corr) < 1e-10
    assert rel_err(gm8.cpu().numpy(), m8) < 1e-10


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


@pytest.mark.parametrize("n_max", [0, 1, 7, 8, 15, 16, 23, 31, 32, 47, 48, 50])
@pytest.mark.parametrize("nz, truncate", [(1, False), (2, False), (1, True)])
def test_edge_correction_by_the_toeplitz_recursion(gpu, orc, nz, truncate, n_max):
    """Diagonally dominant systems of no symmetry take the recursion; one whose leading entry is small,
    one that is nearly singular (pivoted elimination) and a singular one are among them."""
    nb, D = 3, 2 * n_max + 1
    rng = np.random.default_rng(n_max + 100 * nz)
    c = lambda *s: rng.normal(size=s) + 1j * rng.normal(size=s)  # noqa: E731
    norm = c(nz ** 3, D, nb, nb)
    norm[:, 0] = 4.0 * D + rng.normal(size=(nz ** 3, nb, nb))
    norm[0, 0, 0, 1] = norm[0, 0, 1, 0] = 1e-3
    if n_max > 0:
        norm[0, :, 1, 1] = 1.0  # constant in the order: rank one, up to a small diagonal
        norm[0, 0, 1, 1] = 1.0 + 1e-5
    norm[0, :, 2, 2] = 0.0
    ups = c(nz ** 3, 4, n_max + 1, nb, nb)
    setup = dict(n_bins=nb, theta_min=0.7, theta_max=9.0, n_max=n_max, n_z=nz, norm_truncate=truncate)
    want, ns = orc.edge_correct(orc.Setup(**setup), ups, norm)
    with gpu.Estimator(**setup, precision="fp64") as est:
        got, gs = est.edge_correct(torch.as_tensor(ups, device="cuda"), torch.as_tensor(norm, device="cuda"))
    got = got.cpu().numpy()
    assert gs == ns and ns >= 1
    np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
    for b1 in range(nb):
        for b2 in range(nb):
            g, w = got[..., b1, b2], want[..., b1, b2]
            ok = ~np.isnan(w)
            # the nearly singular system: conditioned like D 1e5
            assert rel_err(g[ok], w[ok]) < (1e-8 if b1 == b2 == 1 else 1e-10), (b1, b2)
