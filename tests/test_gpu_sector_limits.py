"""The sector form of the moments (csrc/moments_far.cu) at the limits of its plan: binnings, fields and
orders at the edge of what a context accepts. Pair counts are whole numbers and equal to the FP64 form's
(which has no sectors). Tolerances, normwise against FP64: 1e-4 for gradients, the differentiation form's in
FP32; moments of sector bins 1e-5 (a direction in FP32 is off by at most 1.5 2^-24, an order m <= 100 by m times
that, 9e-6; the dropped Chebyshev terms add 3e-8)."""
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


@pytest.mark.parametrize("n_max, lo, bins", [(50, 200.0, 2), (45, 200.0, 4)])
def test_first_bin_hundreds_of_cells_away(gpu, n_max, lo, bins):
    """8.6 galaxies per arcmin^2, bins from 200' (590 cells) up, half of the patch with few centres, so that
    groups extend over all the rows and columns allowed: cells and groups must be as narrow as the expansion in
    the angle from a sector's axis assumes. One galaxy of every bin carries weight, near the y axis (a sector's
    boundary) as seen from the groups, so each moment is that galaxy's phase and an error of its direction
    shows in full."""
    rng = np.random.default_rng(n_max)
    width, height = 60.0, 860.0
    n = int(8.6 * width * height)
    xy = rng.uniform(0, 1, (n, 2)) * [width, height]
    with gpu.Estimator(bins, lo, 400.0, n_max) as est:
        edges, _ = est.bin_edges()
    cat = hand_catalog(xy, 0.3 * np.exp(1j * rng.uniform(0, 2 * np.pi, n)), np.ones(n))
    dev = gpu.catalog_to_device(cat)
    x, y = xy.T
    share = np.where((x > 5) & (x < 25), 0.6, np.where((x > 30) & (x < 50), 0.066, 0.0))
    mask = (np.abs(y - 0.5 * height) < 30.0) & (rng.uniform(size=n) < share)
    mask = torch.as_tensor(mask.astype(np.uint8)).cuda()
    worst = 0.0
    for x0 in (36.5, 43.5):
        w = np.zeros(n, np.float32)
        for i in range(bins):
            at = [x0, 0.5 * height + (-1) ** i * (edges[i] + 33.0)]
            w[np.argmin(np.hypot(*(xy - at).T))] = 1.0
        w = torch.as_tensor(w).cuda()
        out = {}
        for precision in ("fp64", "fp32"):
            with gpu.Estimator(bins, lo, 400.0, n_max, precision=precision) as est:
                est.accumulate_moments(*dev[:4], w, centre_mask=mask)
                out[precision] = [est.counts(), *est.moments()]
        assert out["fp32"][0] == out["fp64"][0]
        for a, b, unit in zip(out["fp32"][1:], out["fp64"][1:], (0.3, 1.0)):
            worst = max(worst, float((a.to(torch.complex128) - b).abs().max()) / unit)
    print(n_max, lo, bins, worst)
    assert worst < 1e-5


def test_line_over_the_whole_extent(gpu):
    """2.2e6 galaxies on a line of 2^24 quanta: without a limit the grid would have 5.6e6 columns, more than
    the FP32 column arithmetic holds. Pair counts of the three forms against sorted positions."""
    rng = np.random.default_rng(8)
    n, q = 2_200_000, 2.0 ** -13
    x = np.sort(rng.integers(0, 2 ** 24 - 1, n)).astype(np.int64)
    x[0], x[-1] = 0, 2 ** 24 - 1
    ones = torch.ones(n).cuda()
    dev = [torch.as_tensor(rng.permutation(x).astype(np.int32)).cuda(), torch.zeros(n, dtype=torch.int32).cuda(), ones, ones, ones]
    for b0, b1 in ((5.0, 21.5), (21.5, 92.8), (92.8, 400.0)):  # narrow, middle and sector bins
        for precision in ("fp32", "fp64"):
            with gpu.Estimator(1, b0 * q, b1 * q, 10, precision=precision, cell_occupancy=1) as est:
                e2 = est.bin_edges()[1]
                lo, hi = (int(np.ceil(np.sqrt(float(e)))) for e in e2)  # dx^2 in [e2_0, e2_1), dx >= lo, dx < hi
                want = 2 * int((np.searchsorted(x, x + hi) - np.searchsorted(x, x + lo)).sum())
                est.accumulate_moments(*dev)
                assert est.counts() == (n, want), (b0, precision)
