"""A batch whose catalogs differ in the forms their bins take (sector bins from some 6000 galaxies up): graph
and direct runs and single calls give the same bits."""
import numpy as np
import pytest

from paper_2309_08601_gb300 import synth

pytestmark = pytest.mark.gpu

TH = [[2.0, 2.0, 2.0], [4.0, 4.0, 4.0]]


@pytest.mark.parametrize("n_z", [1, 2])
@pytest.mark.parametrize("precision", ["bf16x3", "fp64"])
def test_catalogs_of_different_plans(n_z, precision):
    from paper_2309_08601_gb300 import api
    from paper_2309_08601_gb300.build import build_native
    build_native()
    rng = np.random.default_rng(n_z)
    cats, plans = [], set()
    for i, n in enumerate((3000, 20011, 1500, 9000, 6000, 15000)):
        cat = synth.make_catalog(n, 60.0, 10 + i, field="noise", weights="uniform")
        if n_z > 1:
            cat.zbin = rng.integers(0, n_z, n).astype(np.uint8)
        dev = api.catalog_to_device(cat)
        cats.append(dev if n_z > 1 else dev[:5])
    q = int(60.0 / synth.QUANTUM) + 1
    ext = (0, 0, q, q)
    setup = dict(n_bins=9, theta_min=0.5, theta_max=30.0, n_max=12, n_z=n_z, precision=precision)
    with api.Estimator(**setup) as est:
        graphs = est.run_batch(cats, ext, TH, use_graphs=True).cpu().numpy()
        launches, _ = est.graph_stats()
        assert est.last_error() == "" and launches == len(cats) - 1
        direct = est.run_batch(cats, ext, TH, use_graphs=False).cpu().numpy()
    single = []
    with api.Estimator(**setup) as est:
        est.set_extent(ext)
        for c in cats:
            est.stage_times()
            est.accumulate_moments(*c)
            plans.add(est.stage_times()["moments"][1])
            m = est.measure(*c[:5], theta_ap=TH, zbin=c[5] if n_z > 1 else None, report_singular=False)
            single.append(m.m8.cpu().numpy())
    assert len(plans) > 1 or precision == "fp64"
    np.testing.assert_array_equal(graphs, direct)
    np.testing.assert_array_equal(graphs, np.stack(single))
