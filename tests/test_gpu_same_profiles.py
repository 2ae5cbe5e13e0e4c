"""Bands of a fit without random weights (no slip, C0): all trials have one profile."""
import ctypes

import numpy as np
import pytest

from oracle import surrogate as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cfd", [1, 2, 33, 200, 1024, 1025, 3000])
@pytest.mark.parametrize("trials", [1, 2, 3, 100, 257, 1000])
def test_mean_does_not_depend_on_the_deviation(n_cfd, trials):
    """The mean is the same to the bit whether a standard deviation is asked for or not.  Profile:
    sums of n_cfd terms of one sign in binary64 (rounding below n_cfd 2^-53 of the largest value,
    bounded here by 1e-11); deviation: rounding only."""
    from paper_2311_14140_gb300 import Surrogate
    from paper_2311_14140_gb300 import dsmc as D
    Kn, F = 0.2, 8e-3
    raw = D.SurrogateFit()
    raw.sel_v = raw.sel_c = 0
    raw.sigma_p, raw.sigma_p_var = 1.05, 0.01
    for k, b in enumerate(S.exponents(Kn)):
        raw.b[k] = b
    z = np.random.default_rng(7).standard_normal((trials, 4))
    s = Surrogate(Kn, F, 50, 50)
    mean, sd = s.profile(n_cfd, z, {"_raw": raw})
    alone = np.empty(n_cfd)
    D._check(s._lib.dsmc_surrogate_profile(s._h, ctypes.byref(raw), n_cfd, D._ptr(z), trials,
                                           D._ptr(alone), None))
    s.close()
    np.testing.assert_array_equal(alone, mean)
    want = S.cfd(Kn, F, n_cfd, None, (), ())
    scale = np.abs(want).max()
    np.testing.assert_allclose(mean, want, rtol=0, atol=1e-11 * scale)
    assert (sd >= 0.0).all() and sd.max() <= 1e-11 * scale
