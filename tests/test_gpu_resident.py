"""Resident steps (csrc/dsmc_resident.cu) against the span passes, bit for bit.

A handle with default options runs small problems resident, on a cluster of CTAs up to 40,000
particles and on a team of them over the whole device above; with profile=1 the
same handle takes the span passes (whose parity with the oracle the other tests pin).  Both
must give the same records, offsets, maxima, counters and moment sums at the sizes where the
resident kernel's tables and partitions can go wrong.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _bits(a):
    a = np.ascontiguousarray(a)
    return a.view(np.uint8)


def _snapshot(h, i=None):
    args = () if i is None else (i,)
    m, n = h.moments(*args)
    return (*h.state(*args), *h.cells(*args), m, np.int64(n))


def _assert_same(a, b):
    for k, (x, y) in enumerate(zip(a, b)):
        np.testing.assert_array_equal(_bits(x), _bits(y), err_msg=f"output {k}")


CASES = [
    dict(Kn=1.0, n_cells=100, ppc=200, omega=0.5),              # the small hard-sphere run
    dict(Kn=0.1, n_cells=200, ppc=50, omega=0.5),               # the training run
    dict(Kn=0.44, n_cells=45, ppc=50, omega=0.81),              # the hybrid's sub-domain
    dict(Kn=0.5, n_cells=200, ppc=500, omega=0.5),              # largest shares
    dict(Kn=1.0, n_cells=7, ppc=3, omega=1.0),                  # fewer particles than lanes
    dict(Kn=1.0, n_cells=1, ppc=700, omega=0.5),                # one cell over all CTAs
    dict(Kn=10.0, n_cells=37, ppc=533, omega=0.74),             # about one wall hit each
    dict(Kn=0.5, n_cells=3, ppc=5, omega=0.5, group_size=2),    # groups of two
    dict(Kn=0.1, n_cells=20, ppc=3000, omega=0.81, accum=1),    # many groups per cell
    dict(Kn=0.1, n_cells=700, ppc=20, omega=0.5, group_size=8),  # more cells than threads
    dict(Kn=0.3, n_cells=300, ppc=100, omega=0.5, collisions=False),
    dict(Kn=0.3, n_cells=60, ppc=300, omega=0.81, group_size=512),
    dict(Kn=0.3, n_cells=400, ppc=103, omega=0.81),             # the smallest team runs
    dict(Kn=0.3, n_cells=1, ppc=50000, omega=0.5),              # one cell over a team
    dict(Kn=5.0, n_cells=37, ppc=2000, omega=1.0, accum=1),     # fewer cells than CTAs
    dict(Kn=0.1, n_cells=1200, ppc=50, omega=0.5, group_size=64),  # more cells than threads
    dict(Kn=0.3, n_cells=397, ppc=2531, omega=0.81),            # a full device
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c['n_cells']}x{c['ppc']}")
def test_resident_steps_match_the_span_passes(case):
    from paper_2311_14140_gb300 import Dsmc
    got = []
    for profile in (False, True):
        d = Dsmc(body_force=1e-2, seed=5, sample_start=4, profile=profile, **case)
        for n in (1, 2, 7, 3):  # odd and even counts: every buffer parity
            d.step(n)
        got.append(_snapshot(d))
        d.close()
    _assert_same(*got)


@pytest.mark.parametrize("ppc", [150, 1500])
def test_resident_steps_of_an_uneven_state_and_open_boundary(ppc):
    """A loaded state that fills only part of the channel (empty cells, dense cells), then
    an open upper boundary; switching between the two step kinds on the way."""
    from paper_2311_14140_gb300 import Dsmc
    rng = np.random.default_rng(3)
    n = 60 * ppc
    y = (0.35 * rng.random(n) ** 2 + 0.5).astype(np.float32)
    v = [rng.normal(0, np.sqrt(0.5), n).astype(np.float32) for _ in range(3)]
    got = []
    for profile in (False, True):
        d = Dsmc(0.3, 60, ppc, omega=0.81, body_force=1e-2, seed=9, profile=profile)
        d.load_state(y, *v, step=3)
        d.step(4)
        d.set_open_top(0.01, -0.02)
        d.step(5)
        d.set_options(profile=not profile)
        d.step(2)
        d.set_options(profile=profile)
        d.step(3)
        got.append(_snapshot(d))
        d.close()
    _assert_same(*got)


@pytest.mark.parametrize("n,cells,ppc", [(2, 30, 41), (9, 0, 0), (40, 100, 100), (24, 200, 200)])
def test_resident_batches_match_the_span_passes(n, cells, ppc):
    from paper_2311_14140_gb300 import DsmcBatch
    defs = [dict(Kn=0.2 + 0.3 * i, n_cells=cells or 30 + 7 * i, ppc=ppc or 40 + 11 * i,
                 omega=(0.5, 0.81, 1.0)[i % 3], body_force=1e-3, seed=i) for i in range(n)]
    got = []
    for profile in (False, True):
        b = DsmcBatch(defs, sample_start=3, profile=profile)
        b.step(5)
        b.step(6)
        got.append([_snapshot(b, i) for i in range(n)])
        b.close()
    for a, b in zip(*got):
        _assert_same(a, b)


@pytest.mark.parametrize("n_cells,ppc,group_size", [(60, 3, 256), (40, 50, 256), (30, 500, 512),
                                                    (6, 25000, 256)])
def test_error_keeping_sums_of_known_velocities(n_cells, ppc, group_size):
    """accum=1 without collisions: the sums before and after the collisions are those of the
    state before the step, so a step's moments are known exactly (math.fsum of the binary32
    products).  Bound: every group total is rounded to its cell's grid (half a step of
    2^-(41 - e) per group, e the bit length of the cell's count) after an addition error of at
    most 2^-40 of the sum of |products|, halved and doubled again by the two samples."""
    import math

    from paper_2311_14140_gb300 import Dsmc
    d = Dsmc(0.1, n_cells, ppc, omega=0.81, body_force=1e-3, seed=3, accum=1, collisions=False,
             group_size=group_size, sample_start=2)
    d.step(1)
    _, x, y, z = d.state()
    off = d.cells()[0]
    d.step(1)
    sums, n = d.moments()
    d.close()
    assert n == 1
    xx, yy, zz = x * x, y * y, z * z
    v2 = (xx + yy) + zz
    prods = [x, y, z, xx, yy, zz, x * y, x * z, y * z, x * v2, y * v2, z * v2]
    for c in range(n_cells):
        nc = int(off[c + 1] - off[c])
        groups = nc // group_size + 1
        grid = 2.0 ** -(41 - nc.bit_length())
        for k, p in enumerate(prods):
            q = p[off[c]:off[c + 1]].astype(np.float64)
            bound = 0.5 * grid * groups + 2.0 ** -40 * np.abs(q).sum()
            assert abs(sums[c, k + 1] - math.fsum(q)) <= bound, (c, k)
