"""The adjoint of the contraction at the edges of its tiles: one bin and 64 (the staged table and rows
single, several passes of the threads), odd bin counts, tomographic bins, one centre more or less than a
tile of 64.

L = Re sum conj(gu) Upsilon + conj(gn) N with random gu, gn is a cubic in the shears and a cubic in
the weights, so D(h) = (L(x + h d) - L(x - h d)) / 2h has (4 D(h) - D(2h)) / 3 as its exact slope.
Shears, weights, directions and steps are multiples of 2^-10 and exact in float32, L comes from the
FP64 form. Tolerances, relative to sum |gradient . direction|: the FP64 gradients are returned in
float32, 2^-24 a term, so 2e-7; FP32 1e-4 as in the other tests of the differentiation form.
"""
import numpy as np
import pytest
import torch

from tests._util import hand_catalog

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bins,n_max,n_z,centres", [(1, 1, 1, 64), (7, 4, 2, 65), (20, 5, 1, 63), (33, 3, 3, 130),
                                                      (64, 2, 2, 129)])
def test_contraction_adjoint_tiles(n_bins, n_max, n_z, centres):
    from paper_2309_08601_gb300 import api
    from paper_2309_08601_gb300.build import build_native
    build_native()
    rng = np.random.default_rng(n_bins)
    n = 190
    q = 2.0 ** -10
    zb = rng.integers(0, n_z, n) if n_z > 1 else None
    cat = hand_catalog(rng.uniform(0, 9, (n, 2)), np.zeros(n), np.ones(n), zbin=zb)
    xq, yq, _, _, _, z = api.catalog_to_device(cat)
    g = [torch.as_tensor(q * rng.integers(-400, 400, n), dtype=torch.float32).cuda() for _ in range(2)]
    w = torch.as_tensor(q * rng.integers(512, 1536, n), dtype=torch.float32).cuda()
    mask = torch.zeros(n, dtype=torch.uint8)
    mask[torch.as_tensor(rng.permutation(n)[:centres])] = 1
    mask = mask.cuda()
    setup = dict(n_bins=n_bins, theta_min=0.3, theta_max=8.0, n_max=n_max, n_z=n_z)

    with api.Estimator(**setup, precision="fp64") as e64:
        ups, norm = e64.new_multipoles()
        gu, gn = (torch.complex(*[torch.as_tensor(rng.normal(size=tuple(t.shape))) for _ in range(2)]).cuda()
                  for t in (ups, norm))

        def value(a, b, c):
            e64.accumulate_moments(xq, yq, a, b, c, z, mask)
            u, m = e64.contract()
            return float((gu.conj() * u).sum().real + (gn.conj() * m).sum().real)

        def slope(dirs):
            def d(h):
                p, m = ([x + s * h * y for x, y in zip((*g, w), dirs)] for s in (1, -1))
                return (value(*p) - value(*m)) / (2 * h)
            return (4 * d(0.125) - d(0.25)) / 3

        zero = torch.zeros_like(w)
        rnd = lambda: torch.as_tensor(8 * q * rng.integers(-64, 64, n), dtype=torch.float32).cuda()
        dirs = [(rnd(), rnd(), zero), (zero, zero, rnd())]
        want = [slope(d) for d in dirs]
        for precision, tol in (("fp64", 2e-7), ("fp32", 1e-4)):
            with api.Estimator(**setup, precision=precision) as est:
                est.accumulate_moments(xq, yq, *g, w, z, mask)
                grad = [t.double() for t in est.moments_adjoint(gu, gn, *g, w)]
            for d, v in zip(dirs, want):
                terms = sum(x * y.double() for x, y in zip(grad, d))
                assert abs(float(terms.sum()) - v) < tol * float(terms.abs().sum()), (precision, float(terms.sum()), v)
