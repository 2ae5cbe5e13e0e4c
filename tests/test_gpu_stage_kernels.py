"""The surrogate stage's kernels at the edges of their chunks and tiles, against the oracle.

Tolerances: the CFD profiles are sums of n terms of one sign pattern in binary64 (rounding of
about n 2^-53 of the largest value, bounded here by 1e-11)."""
import numpy as np
import pytest

from oracle import surrogate as S

pytestmark = pytest.mark.gpu


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
