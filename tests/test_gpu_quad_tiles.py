"""Tensor-core contraction with four sides per tile (up to 16 bins): orders that fill a tile and orders
that end inside one, against the oracle's contraction of the same FP32 moments (2e-5 for BF16x3, 2e-6
for TF32x3: the split products' bounds, as in the other tensor-core tests)."""
import numpy as np
import pytest

from tests._util import hand_catalog, rel_err
from tests.test_gpu_parity import run

pytestmark = pytest.mark.gpu

TOL = {"bf16x3": 2e-5, "tf32x3": 2e-6}


@pytest.fixture(scope="module")
def gpu():
    import torch
    from paper_2309_08601_gb300.build import build_native
    build_native()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2309_08601_gb300 import api
    return api


@pytest.mark.parametrize("precision", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("n_bins, n_max, n_z", [(16, 0, 1), (16, 1, 1), (15, 2, 2), (14, 3, 1), (13, 4, 1), (12, 5, 2),
                                                (9, 6, 1), (8, 7, 1), (2, 3, 3)])
def test_quad_tiles(gpu, orc, precision, n_bins, n_max, n_z):
    rng = np.random.default_rng(10 * n_bins + n_max)
    n = 900
    cat = hand_catalog(rng.uniform(0, 18, (n, 2)), rng.normal(0, .3, n) + 1j * rng.normal(0, .3, n),
                       rng.uniform(0.5, 1.5, n), rng.integers(0, n_z, n) if n_z > 1 else None)
    setup = dict(n_bins=n_bins, theta_min=0.3, theta_max=9.0, n_max=n_max, n_z=n_z)
    g = run(gpu, cat, setup, precision, theta=[[1.0, 1.0, 1.0]])
    ups, norm = orc.contract(orc.Setup(**setup), cat, g["G"].astype(np.complex128), g["W"].astype(np.complex128))
    assert rel_err(g["ups"], ups) < TOL[precision]
    assert rel_err(g["norm"], norm) < TOL[precision]
