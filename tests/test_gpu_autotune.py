"""dsmc_autotune and the option changes after it: the tuner's partition is not the caller's."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

SMALL = [dict(Kn=0.2 + 0.1 * i, n_cells=100, ppc=100, body_force=1e-3, seed=i) for i in range(12)]
FEW_CELLS = [dict(Kn=0.3, n_cells=60, ppc=40000, omega=0.81, body_force=1e-3, seed=1)]
SPLIT = ("span_particles", "cta_warps", "span_rows", "cells_per_span", "n_spans", "total_spans")


def _split(b):
    return {k: b.info(0)[k] for k in SPLIT}


def _kind(b):
    b.step(2)
    return b.last_step()[0]


def test_tuned_batch_keeps_its_kind_of_steps():
    from paper_2311_14140_gb300 import DsmcBatch
    b = DsmcBatch(SMALL)
    assert _kind(b) == "clusters"
    b.autotune(steps_per_trial=1)
    split = _split(b)
    assert _kind(b) == "clusters"
    b.set_options(sample_start=50)  # gives the tuner's values back
    assert _kind(b) == "clusters"
    assert _split(b) == split
    b.set_options(span_particles=2 * split["span_particles"])  # named by the caller
    assert _kind(b) == "spans"
    b.set_options(sample_start=60)
    assert _kind(b) == "spans"
    b.set_options(span_particles=0, cta_warps=0, span_rows=0)
    assert _kind(b) == "clusters"
    b.close()


def test_partition_named_before_tuning_stays_named():
    from paper_2311_14140_gb300 import DsmcBatch
    b = DsmcBatch(SMALL, cta_warps=4)
    assert _kind(b) == "spans"
    b.autotune(steps_per_trial=1)
    b.set_options(sample_start=50)
    assert _kind(b) == "spans"
    b.close()


def test_tuner_returns_the_partition_that_is_kept():
    """60 cells of 40,000 particles: several CTAs share a cell unless a partition is named."""
    from paper_2311_14140_gb300 import DsmcBatch
    b = DsmcBatch(FEW_CELLS)
    assert b.info(0)["n_spans"] > 60
    best, ms = b.autotune(steps_per_trial=3)
    split = _split(b)
    assert best == split["span_particles"] and ms > 0
    b.set_options(sample_start=5)
    assert _split(b) == split
    b.set_options(span_particles=4096 if best != 4096 else 8192)
    assert b.info(0)["n_spans"] <= 60  # whole cells
    b.close()


def test_named_shape_leaves_whole_cells():
    """Naming the CTA shape alone takes the partition out of the library's hands too."""
    from paper_2311_14140_gb300 import DsmcBatch
    b = DsmcBatch(FEW_CELLS)
    b.set_options(cta_warps=4)
    assert b.info(0)["n_spans"] <= 60
    b.close()


@pytest.mark.parametrize("defs", [SMALL, FEW_CELLS], ids=["batch", "few_cells"])
def test_failed_tuning_leaves_the_partition(defs):
    """Trials cannot be timed while the stream is being captured: the tuner reports that, and the
    handle has the partition from before."""
    import torch

    from paper_2311_14140_gb300 import DsmcBatch, DsmcError
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        b = DsmcBatch(defs, stream=stream.cuda_stream)
        b.step(2)
        b.sync()
        before = _split(b)
        s, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
        relaxed = 2
        assert cu.cuStreamBeginCapture_v2(s, relaxed) == 0
        try:
            with pytest.raises(DsmcError):
                b.autotune(steps_per_trial=1)
        finally:
            cu.cuStreamEndCapture(s, ctypes.byref(graph))
        if graph:
            cu.cuGraphDestroy(graph)
        assert _split(b) == before
        b.close()
    # nothing of the failure is left for the next call
    c = DsmcBatch(SMALL)
    c.step(2)
    c.sync()
    c.close()
