"""Span passes whose cells are shared by several CTAs (one run with few, populous cells) against
the same passes with whole-cell spans (a named partition), bit for bit; profile=1 keeps both off
the resident path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _bits(a):
    return np.ascontiguousarray(a).view(np.uint8)


def _same(runs):
    out = []
    for d in runs:
        m, n = d.moments()
        out.append((*d.state(), *d.cells(), m, np.int64(n)))
    for k, (x, y) in enumerate(zip(*out)):
        np.testing.assert_array_equal(_bits(x), _bits(y), err_msg=f"output {k}")


@pytest.mark.parametrize("case", [
    dict(Kn=0.5, n_cells=1, ppc=50000, omega=0.5),                 # one cell in 13 shares
    dict(Kn=0.3, n_cells=7, ppc=30011, omega=0.81, accum=1),
    dict(Kn=5.0, n_cells=20, ppc=9001, omega=0.74, group_size=512),  # many wall hits
    dict(Kn=0.3, n_cells=300, ppc=6000, omega=1.0),                # two shares per cell
    dict(Kn=0.3, n_cells=3, ppc=7000, omega=0.5, collisions=False),
    dict(Kn=0.3, n_cells=40, ppc=40000, omega=0.81),               # beyond the resident sizes
])
def test_shared_cells_match_whole_cell_spans(case):
    from paper_2311_14140_gb300 import Dsmc
    a = Dsmc(body_force=1e-2, seed=5, sample_start=3, profile=True, **case)
    b = Dsmc(body_force=1e-2, seed=5, sample_start=3, profile=True, span_particles=4096, **case)
    assert a.info()["n_spans"] > case["n_cells"] and b.info()["n_spans"] == case["n_cells"]
    for d in (a, b):
        d.step(3)
        d.step(4)
    _same((a, b))
    a.reset_samples()
    b.reset_samples()
    a.set_options(span_rows=2)
    for d in (a, b):
        d.step(3)
    _same((a, b))
    a.close()
    b.close()


def test_shared_cells_of_an_uneven_state():
    """A loaded state that leaves cells empty and others with fewer groups than shares."""
    from paper_2311_14140_gb300 import Dsmc
    rng = np.random.default_rng(2)
    n = 12 * 20000
    y = (0.3 * rng.random(n) ** 3 + 0.6).astype(np.float32)
    y[:3] = 0.01
    v = [rng.normal(0, np.sqrt(0.5), n).astype(np.float32) for _ in range(3)]
    runs = [Dsmc(0.3, 12, 20000, omega=0.81, body_force=1e-2, seed=9, profile=True, **kw)
            for kw in ({}, dict(span_particles=4096))]
    for d in runs:
        d.load_state(y, *v, step=3)
        d.step(5)
    _same(runs)


def test_shared_cells_under_graph_replay():
    import torch

    from paper_2311_14140_gb300 import Dsmc
    s = torch.cuda.Stream()
    runs = [Dsmc(0.3, 40, 40000, omega=0.81, body_force=1e-2, seed=9, sample_start=5, graph=g,
                 stream=s.cuda_stream) for g in (True, False)]
    for d in runs:
        d.step(37)
    _same(runs)


def test_cells_that_fill_a_wave_stay_whole():
    """Both ends of the range of cell counts whose whole cells fill three CTAs per SM."""
    import torch

    from paper_2311_14140_gb300 import Dsmc
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lo, hi = -(-12 * sms // 5), 3 * sms
    for n, whole in ((lo - 1, False), (lo, True), (hi, True), (hi + 1, False)):
        kw = dict(Kn=0.3, n_cells=n, ppc=10000, omega=0.81, seed=4, profile=True)
        runs = [Dsmc(**kw), Dsmc(span_particles=4096, **kw)]
        assert (runs[0].info()["n_spans"] == n) is whole
        for d in runs:
            d.step(2)
        _same(runs)
        for d in runs:
            d.close()
