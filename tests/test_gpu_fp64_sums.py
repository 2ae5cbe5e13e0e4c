"""DSMC_ACCUM_FP64 keeps at least the bits of binary64 additions.

Velocities of magnitudes spread over 2^14 make products whose sums need more than 48 bits.  The
moment sums of one step without collisions (every particle counted before and after them) are
compared with exact sums of the binary32 products.  Bound per cell and moment, for one group of n
particles: binary64 additions of 2 ceil(n / 32) products per lane and over 32 lanes lose at most
(2 ceil(n / 32) + 5) 2^-53 of the sum of |products|, the rounding to the cell's grid 2^-(41 - e), e
the bit length of n, half a grid step, and the conversion to binary64 2^-53 of the total."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N_CELLS = 8


def _products(v):
    x, y, z = v
    v2 = (x * x + y * y) + z * z
    return [x, y, z, x * x, y * y, z * z, x * y, x * z, y * z, x * v2, y * v2, z * v2]


@pytest.mark.parametrize("spans", [True, False])
@pytest.mark.parametrize("ppc,group", [(7, 256), (31, 256), (63, 256), (200, 256), (383, 256),
                                       (767, 512)])
def test_sums_keep_the_bits_of_binary64(ppc, group, spans):
    from paper_2311_14140_gb300 import Dsmc
    rng = np.random.default_rng(ppc)
    n = N_CELLS * ppc
    v = (np.exp2(rng.uniform(-8.0, 5.8, (3, n))) * rng.choice([-1, 1], (3, n))).astype(np.float32)
    y = ((np.repeat(np.arange(N_CELLS), ppc) + 0.5) / N_CELLS).astype(np.float32)
    d = Dsmc(0.5, N_CELLS, ppc, omega=0.81, dt=1e-4, collisions=False, group_size=group, accum=1,
             seed=1, span_particles=1024 if spans else 0)
    d.load_state(y, *v, step=0)
    d.step(1)
    acc, steps = d.moments()
    d.close()
    assert steps == 1
    for c in range(N_CELLS):
        cell = [p[c * ppc:(c + 1) * ppc] for p in _products(v)]
        assert acc[c, 0] == ppc
        for k, p in enumerate(cell):
            assert p.dtype == np.float32
            exact = math.fsum(map(float, p))  # half of before plus after
            mag = math.fsum(abs(float(t)) for t in p)
            bound = ((2 * -(-ppc // 32) + 5) * 2.0 ** -53 * mag + 2.0 ** -53 * abs(exact)
                     + 0.25 * 2.0 ** -(41 - ppc.bit_length()))
            assert abs(acc[c, k + 1] - exact) <= bound, (c, k)
