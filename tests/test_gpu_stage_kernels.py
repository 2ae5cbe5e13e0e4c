"""The surrogate stage's kernels at the edges of their chunks and tiles, against the oracle.

Tolerances: the CFD profiles are sums of n terms of one sign pattern in binary64 (rounding of
about n 2^-53 of the largest value, bounded here by 1e-11); the GP's marginal likelihoods and
predictions as in the tests of the larger designs."""
import numpy as np
import pytest

from oracle import gp as GP
from oracle import surrogate as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 255, 256, 257, 1000])
def test_face_cfd_sizes(n):
    from paper_2311_14140_gb300 import cfd_faces
    Kn, F = 0.3, 5e-3
    Sf = S.stress_correction(np.arange(n + 1) / n, (0.3, -0.1), S.exponents(Kn)[:2])
    for sp in (None, 1.1):
        want = GP.cfd_faces(Kn, F, n, sp, Sf)
        np.testing.assert_allclose(cfd_faces(Kn, F, n, sp, Sf), want, rtol=0,
                                   atol=1e-11 * np.abs(want).max())


@pytest.mark.parametrize("n_cfd,trials", [(1, 2), (2, 1), (33, 255), (256, 257), (257, 256),
                                          (700, 3)])
@pytest.mark.parametrize("k", [0, 1, 3])
def test_bands_of_a_given_fit(n_cfd, trials, k):
    """Bands of a fit given outright (k correction weights, slip for odd k) against the
    trials' profiles solved one by one."""
    from paper_2311_14140_gb300 import Surrogate
    from paper_2311_14140_gb300 import dsmc as D
    Kn, F = 0.2, 8e-3
    b = S.exponents(Kn)
    raw = D.SurrogateFit()
    raw.sel_v, raw.sel_c = k % 2, k
    raw.sigma_p, raw.sigma_p_var = 1.05, 0.01
    m = np.array([0.02, -0.01, 0.005])[:k]
    A = np.random.default_rng(k).normal(size=(3, 3))[:k, :k]
    cov = 1e-4 * (A @ A.T + np.eye(k))
    for i in range(k):
        raw.m_c[k][i] = m[i]
        for j in range(k):
            raw.S_c[k][3 * i + j] = cov[i, j]
    for l in range(3):
        raw.b[l] = b[l]
    z = np.random.default_rng(7).standard_normal((trials, 4))
    mean, sd = Surrogate(Kn, F, 50, 50).profile(n_cfd, z, {"_raw": raw})
    w = m + z[:, 1:1 + k] @ np.linalg.cholesky(cov).T if k else np.zeros((trials, 0))
    prof = np.array([S.cfd(Kn, F, n_cfd, 1.05 + 0.1 * z[t, 0] if k % 2 else None, tuple(w[t]),
                           b[:k]) for t in range(trials)])
    scale = np.abs(prof).max()
    np.testing.assert_allclose(mean, prof.mean(axis=0), rtol=0, atol=1e-11 * scale)
    want = prof.std(axis=0, ddof=1) if trials > 1 else np.zeros(n_cfd)
    np.testing.assert_allclose(sd, want, rtol=0, atol=1e-11 * scale)


@pytest.mark.parametrize("n,m", [(2, 1), (3, 7), (17, 8), (33, 9), (127, 3), (128, 40)])
def test_gp_sizes(n, m):
    from paper_2311_14140_gb300 import GaussianProcess
    rng = np.random.default_rng(n)
    X = rng.uniform(size=(n, 2))
    Y = np.sin(3 * X[:, :1]) * np.linspace(0.5, 2, m) + 0.1 * rng.normal(size=(n, m))
    g = GaussianProcess(X, Y, GP.GRID)
    o = GP.fit(X, Y)
    np.testing.assert_allclose(g.lml, o["lml"], rtol=1e-9, atol=1e-9 * n * m)
    assert g.best == o["best"]
    Xs = rng.uniform(size=(5, 2))
    np.testing.assert_allclose(g.predict(Xs), GP.predict(o, Xs), rtol=1e-8,
                               atol=1e-10 * np.abs(Y).max())


def test_gp_grid_larger_than_one_chunk():
    """6,001 hyperparameter points of 64-point factors take more than one chunk; the chosen
    point lies in the first, so its factor is formed again."""
    from paper_2311_14140_gb300 import GaussianProcess
    rng = np.random.default_rng(1)
    X = rng.uniform(size=(64, 2))
    Y = np.sin(3 * X[:, :1]) + 0.1 * rng.normal(size=(64, 2))
    grid = [(0.4, 1.0, 1e-2)] + [(0.05, 0.05, 0.3 + 1e-4 * i) for i in range(6000)]
    g = GaussianProcess(X, Y, grid)
    o = GP.fit(X, Y, grid[:3])
    assert g.best == o["best"]
    Xs = rng.uniform(size=(5, 2))
    np.testing.assert_allclose(g.predict(Xs), GP.predict(o, Xs), rtol=1e-8, atol=1e-10)
