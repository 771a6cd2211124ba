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


def _solve_extended(A, Y):
    """Gaussian elimination with partial pivoting in numpy's extended precision."""
    A, X = A.astype(np.clongdouble), Y.astype(np.clongdouble)
    n = len(A)
    for k in range(n):
        p = k + np.argmax(np.abs(A[k:, k]))
        A[[k, p]], X[[k, p]] = A[[p, k]], X[[p, k]]
        f = A[k + 1:, k] / A[k, k]
        A[k + 1:] -= f[:, None] * A[k]
        X[k + 1:] -= f[:, None] * X[k]
    for k in range(n - 1, -1, -1):
        X[k] = (X[k] - A[k, k + 1:] @ X[k + 1:]) / A[k, k]
    return X


@pytest.mark.parametrize("n_max, kind, par", [(30, "gap", 0.3), (30, "gap", 0.4), (10, "gap", 0.8), (30, "gauss", 1.1),
                                              (30, "few", 75), (30, "few", 3000)])
def test_concentrated_angles(gpu, n_max, kind, par):
    """Couplings sum_j w_j e^{i m phi_j} of angles with a gap, around one direction, or few of them: those conditioned
    1e4 D and worse (the recursion takes systems whose inverse grows by at most 1e4) are solved by the elimination,
    bit for bit. (Times 2^495, where |N_0|^2 leaves the recursion's range, every system is; a power of two changes no
    rounding.) The others, against extended precision: growth D 2^-53, 1e-10, and 1e-13 for many angles (growth 6)."""
    nb, D = 5, 2 * n_max + 1
    rng = np.random.default_rng(D + int(10 * par))
    m = np.arange(D)
    norm = np.zeros((1, D, nb, nb), complex)
    for b1 in range(nb):
        for b2 in range(b1, nb):
            k = 300 if kind == "gauss" else 2000 if kind == "gap" else int(par)
            phi = rng.normal(0, par, k) if kind == "gauss" else rng.uniform(-np.pi + par, np.pi - par, k) if kind == "gap" \
                else rng.uniform(-np.pi, np.pi, k)
            t = (rng.uniform(0.5, 1.5, k) * np.exp(1j * m[:, None] * phi)).sum(1)
            norm[0, :, b1, b2] = t if b1 != b2 else t.real
            norm[0, :, b2, b1] = t.conj() if b1 != b2 else t.real
    ups = rng.normal(size=(1, 4, n_max + 1, nb, nb)) + 1j * rng.normal(size=(1, 4, n_max + 1, nb, nb))
    setup = dict(n_bins=nb, theta_min=0.7, theta_max=9.0, n_max=n_max)
    with gpu.Estimator(**setup, precision="fp64") as est:
        got, scaled = ([est.edge_correct(torch.as_tensor(ups * f, device="cuda"), torch.as_tensor(norm * f, device="cuda"))
                        for f in (1.0, 2.0 ** 495)])
    assert got[1] == scaled[1] == 0
    got, scaled = got[0].cpu().numpy(), scaled[0].cpu().numpy()
    for b1 in range(nb):
        for b2 in range(nb):
            T = lambda d: norm[0, d, b1, b2] if d >= 0 else norm[0, -d, b2, b1]  # noqa: E731
            A = np.array([[T(i - j) for j in range(D)] for i in range(D)])
            if np.linalg.cond(A) > 1e4 * D:
                np.testing.assert_array_equal(got[..., b1, b2], scaled[..., b1, b2])
                continue
            Y = np.array([[ups[0, mu, l, b1, b2] if l >= 0 else ups[0, (0, 1, 3, 2)[mu], -l, b2, b1] for mu in range(4)]
                          for l in range(-n_max, n_max + 1)])
            X = _solve_extended(A, Y)
            assert np.abs(got[0, :, :, b1, b2].T - X).max() < (1e-13 if par == 3000 else 1e-10) * np.abs(X).max()
