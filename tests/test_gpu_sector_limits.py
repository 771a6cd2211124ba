"""The sector form of the moments (csrc/moments_far.cu) at the limits of its plan: binnings, fields and
orders at the edge of what a context accepts. Pair counts are whole numbers and equal to the FP64 form's
(which has no sectors). Tolerances, normwise against FP64: 1e-4 for gradients, the differentiation form's in
FP32."""
import numpy as np
import pytest
import torch

from tests._util import hand_catalog, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    from paper_2309_08601_gb300.build import build_native
    build_native()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2309_08601_gb300 import api
    return api


def _random_gradient(est, seed):
    ups, norm = est.new_multipoles()
    rng = np.random.default_rng(seed)
    return [torch.complex(*[torch.as_tensor(rng.normal(size=tuple(t.shape))) for _ in range(2)]).cuda()
            for t in (ups, norm)]


def test_a_bin_wider_than_any_extent(gpu):
    """theta_max = 1.02e8 quanta, six times the largest extent: no entry of the sorted catalog but the galaxies
    themselves may count as a member, in the sums or in their adjoint."""
    rng = np.random.default_rng(1)
    n, side = 6000, 1000.0
    cat = hand_catalog(rng.uniform(0, side, (n, 2)), 0.3 * (rng.normal(size=n) + 1j * rng.normal(size=n)),
                       rng.uniform(0.5, 1.5, n))
    dev = gpu.catalog_to_device(cat)
    out = {}
    for precision in ("fp64", "fp32"):
        with gpu.Estimator(2, 100.0, 12500.0, 10, precision=precision) as est:
            est.accumulate_moments(*dev)
            out[precision] = [est.counts()]
            gu, gn = _random_gradient(est, 2)
            est.stage_times()
            out[precision] += [t.cpu().numpy() for t in est.moments_adjoint(gu, gn, *dev[2:5])]
            assert (est.stage_times()["moments"][1] > 4) == (precision == "fp32")  # the sector form ran
    assert out["fp32"][0] == out["fp64"][0]
    for a, b in zip(out["fp32"][1:], out["fp64"][1:]):
        assert rel_err(a, b) < 1e-4
