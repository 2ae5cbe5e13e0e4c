"""Which way the steps of a handle take (dsmc_last_step), by sizes and options: the tests that
compare the ways with one another compare nothing where both handles take the same one."""
import pytest

pytestmark = pytest.mark.gpu


def _kind(d):
    assert d.last_step() == (None, 0)
    d.step(2)
    kind = d.last_step()
    d.sync()
    d.close()
    return kind


@pytest.mark.parametrize("n_cells,ppc,opts,kind", [
    (7, 3, {}, "clusters"),
    (100, 200, {}, "clusters"),
    (100, 200, dict(accum=1), "clusters"),
    (1, 700, {}, "clusters"),
    (700, 20, dict(group_size=8), "clusters"),
    (200, 200, {}, "clusters"),   # 40,000: the largest on a cluster
    (271, 148, {}, "team"),       # 40,108
    (1, 50000, {}, "team"),
    (1200, 50, dict(group_size=64), "team"),
    (37, 2000, dict(accum=1), "team"),
    (397, 2531, {}, "team"),
    (400, 3000, {}, "team"),      # 1,200,000
    (400, 4000, {}, "spans"),     # 1,600,000: more than the SMs' shared memory holds
    (16384, 3, {}, "spans"),      # too many cells for a CTA's tables
    (100, 200, dict(profile=True), "spans"),
    (100, 200, dict(span_particles=2048), "spans"),
    (100, 200, dict(cta_warps=4), "spans"),
    (397, 2531, dict(span_rows=2), "spans"),
])
def test_kind_of_one_run(n_cells, ppc, opts, kind):
    from paper_2311_14140_gb300 import Dsmc
    got, ctas = _kind(Dsmc(0.3, n_cells, ppc, omega=0.81, body_force=1e-3, seed=1, **opts))
    assert got == kind
    assert (ctas == 0) == (kind == "spans")


@pytest.mark.parametrize("n,cells,ppc,opts,kind", [
    (2, 30, 41, {}, "clusters"),
    (40, 100, 100, {}, "clusters"),
    (64, 100, 200, {}, "clusters"),
    (24, 200, 200, {}, "clusters"),
    (24, 200, 500, {}, "spans"),
    (256, 100, 200, {}, "spans"),
    (40, 100, 100, dict(cta_warps=4), "spans"),
    (40, 100, 100, dict(profile=True), "spans"),
])
def test_kind_of_a_batch(n, cells, ppc, opts, kind):
    from paper_2311_14140_gb300 import DsmcBatch
    defs = [dict(Kn=0.3 + 0.1 * i, n_cells=cells, ppc=ppc, body_force=1e-3, seed=i)
            for i in range(n)]
    got, ctas = _kind(DsmcBatch(defs, **opts))
    assert got == kind
    assert (ctas == 0) == (kind == "spans")


def test_kind_of_a_pool():
    from paper_2311_14140_gb300 import DsmcPool
    p = DsmcPool(100_000, 400, 4, 200)
    p.add(Kn=0.3, n_cells=100, ppc=200, body_force=1e-3, seed=1)
    p.step(2)
    assert p.last_step() == ("spans", 0)
    p.close()
