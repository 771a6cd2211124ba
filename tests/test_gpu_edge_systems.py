"""Edge-correction systems that the recursion of the FP64 stage must hand to the pivoted elimination, or solve
as accurately as it would."""
import numpy as np
import pytest
import torch

from tests._util import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    from paper_2309_08601_gb300.build import build_native
    build_native()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2309_08601_gb300 import api
    return api


@pytest.mark.parametrize("exponent", [-518, -300, 500])
@pytest.mark.parametrize("n_max", [0, 4])
def test_scaled_systems(gpu, orc, n_max, exponent):
    """Upsilon and N times a power of two: the same Gamma_n (FP64 path, 1e-10), also where |N_0|^2 is denormal."""
    nb, D = 2, 2 * n_max + 1
    rng = np.random.default_rng(n_max)
    c = lambda *s: rng.normal(size=s) + 1j * rng.normal(size=s)  # noqa: E731
    norm, ups = c(1, D, nb, nb), c(1, 4, n_max + 1, nb, nb)
    norm[:, 0] = 4.0 * D
    setup = dict(n_bins=nb, theta_min=0.7, theta_max=9.0, n_max=n_max)
    want, _ = orc.edge_correct(orc.Setup(**setup), ups, norm)
    f = 2.0 ** exponent
    with gpu.Estimator(**setup, precision="fp64") as est:
        got, ns = est.edge_correct(torch.as_tensor(ups * f, device="cuda"), torch.as_tensor(norm * f, device="cuda"))
    assert ns == 0
    assert rel_err(got.cpu().numpy(), want) < 1e-10
