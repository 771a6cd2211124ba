"""The sector form's tables are made by the first call that has sector bins: the same moments as a context
whose first call has them, and a capture that comes first takes the other forms (FP32 path, 1e-4) instead of
allocating."""
import numpy as np
import pytest
import torch

from paper_2309_08601_gb300 import synth
from tests._util import rel_err

pytestmark = pytest.mark.gpu

SETUP = dict(n_bins=8, theta_min=0.5, theta_max=40.0, n_max=12, precision="fp32")


@pytest.fixture(scope="module")
def gpu():
    from paper_2309_08601_gb300.build import build_native
    build_native()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2309_08601_gb300 import api
    return api


@pytest.fixture(scope="module")
def fields(gpu):
    sparse = synth.make_catalog(30_000, 2000.0, 1, field="noise", weights="uniform")
    dense = synth.make_catalog(20_000, 60.0, 2, field="noise", weights="uniform")
    return [gpu.catalog_to_device(c)[:5] for c in (sparse, dense)]


def _launches(est, dev):
    est.stage_times()
    est.accumulate_moments(*dev)
    return est.stage_times()["moments"][1]


def test_tables_on_first_use(gpu, fields):
    sparse, dense = fields
    with gpu.Estimator(**SETUP) as a, gpu.Estimator(**SETUP) as b:
        assert _launches(a, sparse) <= 2  # narrow bins only
        assert _launches(a, dense) == _launches(b, dense) > 4
        for x, y in zip(a.moments(), b.moments()):
            np.testing.assert_array_equal(x.cpu().numpy(), y.cpu().numpy())


def test_capture_before_the_tables(gpu, fields):
    sparse, dense = fields
    ext = lambda side: (0, 0, int(side / synth.QUANTUM) + 1, int(side / synth.QUANTUM) + 1)  # noqa: E731
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        with gpu.Estimator(**SETUP, stream=st) as est, gpu.Estimator(**SETUP, stream=st) as ref:
            est.set_extent(ext(2000.0))
            est.accumulate_moments(*sparse)  # every buffer at its size
            est.set_extent(ext(60.0))
            ref.set_extent(ext(60.0))
            st.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st):
                est.accumulate_moments(*dense)
            for _ in range(2):
                g.replay()
            got = (est.counts(), *est.moments())
            ref.accumulate_moments(*dense)
            want = (ref.counts(), *ref.moments())
            assert got[0] == want[0]
            for x, y in zip(got[1:], want[1:]):
                assert rel_err(x.cpu().numpy(), y.cpu().numpy()) < 1e-4
            del g
