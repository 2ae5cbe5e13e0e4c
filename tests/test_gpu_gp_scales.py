"""Length scales at the ends of the binary64 range: accepted, and answered as by the oracle."""
import numpy as np
import pytest

from oracle import gp as GP

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [5e-324, 1e-310, 2.0 ** -1024, 2.0 ** -1022, 1e-300, 1e300])
@pytest.mark.parametrize("which", [0, 1])
def test_extreme_length_scales(scale, which):
    from paper_2311_14140_gb300 import GaussianProcess
    rng = np.random.default_rng(4)
    X = rng.uniform(size=(20, 2))
    Y = np.sin(3 * X[:, :1]) * np.linspace(0.5, 2, 5) + 0.1 * rng.normal(size=(20, 5))
    point = [0.4, 0.5, 1e-2]
    point[which] = scale
    grid = [tuple(point), (0.4, 0.5, 1e-2)]
    g = GaussianProcess(X, Y, grid)
    with np.errstate(over="ignore"):
        o = GP.fit(X, Y, grid)
    assert np.isfinite(o["lml"]).all()
    np.testing.assert_allclose(g.lml, o["lml"], rtol=1e-9, atol=1e-9 * 20 * 5)
    assert g.best == o["best"]
