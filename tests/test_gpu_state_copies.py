"""dsmc_copy_state / dsmc_load_state with every kind of memory: arrays that kernels can access
(device, pinned host) are written and read in place, all others are copied; the values are the
same.  dsmc_copy_cells into host and device memory."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N_CELLS, PPC = 37, 61  # 2,257 particles: not a multiple of a block


def _run(seed=3):
    from paper_2311_14140_gb300 import Dsmc
    d = Dsmc(0.5, N_CELLS, PPC, omega=0.81, body_force=1e-2, seed=seed)
    d.step(5)
    return d


def _arrays(kind, n):
    import torch
    if kind == "device":
        return [torch.full((n,), np.nan, device="cuda") for _ in range(4)]
    if kind == "pinned":
        return [torch.full((n,), np.nan).pin_memory() for _ in range(4)]
    if kind == "mixed":  # one array of each kind: all are copied
        return [torch.full((n,), np.nan, device="cuda"), torch.full((n,), np.nan).pin_memory(),
                torch.full((n,), np.nan), torch.full((n,), np.nan, device="cuda")]
    if kind == "unaligned":  # byte buffers two past a 4-byte boundary
        return [torch.zeros(4 * n + 2, dtype=torch.uint8, device="cuda")[2:] for _ in range(4)]
    return [torch.full((n,), np.nan) for _ in range(4)]


def _values(t):
    import torch
    t = t.cpu()
    return (t.contiguous().numpy().view(np.uint32) if t.dtype == torch.float32
            else np.frombuffer(t.numpy().tobytes(), np.uint32))


@pytest.mark.parametrize("kind", ["pageable", "pinned", "device", "mixed", "unaligned"])
def test_state_into_and_from(kind):
    d = _run()
    want = [a.view(np.uint32) for a in d.state()]
    got = _arrays(kind, d.N)
    d.state_into(*got)
    for w, g in zip(want, got):
        np.testing.assert_array_equal(_values(g), w)
    part = _arrays(kind, d.N)
    d.state_into(vx=part[1], vz=part[3])  # NULL arrays are left out
    np.testing.assert_array_equal(_values(part[1]), want[1])
    np.testing.assert_array_equal(_values(part[3]), want[3])
    # restored from such arrays, the run goes on as it would have
    e = _run(seed=3)
    e.step(2)
    e.load_state(*got, smax=d.cells()[1], step=5)
    d.step(4)
    e.step(4)
    for a, b in zip(d.state(), e.state()):
        np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))
    d.close()
    e.close()


def test_cells_into_device_memory():
    import torch

    from paper_2311_14140_gb300.dsmc import _check
    d = _run()
    off, smax, ncand, nacc = d.cells()
    t = [torch.zeros(N_CELLS + 1, dtype=torch.int32, device="cuda"),
         torch.zeros(N_CELLS, device="cuda"),
         torch.zeros(N_CELLS, dtype=torch.int64, device="cuda"),
         torch.zeros(N_CELLS, dtype=torch.int64).pin_memory()]
    _check(d._lib.dsmc_copy_cells(d._h, *[ctypes.c_void_p(x.data_ptr()) for x in t]))
    np.testing.assert_array_equal(t[0].cpu().numpy(), off)
    np.testing.assert_array_equal(t[1].cpu().numpy(), smax)
    np.testing.assert_array_equal(t[2].cpu().numpy(), ncand.astype(np.int64))
    np.testing.assert_array_equal(t[3].numpy(), nacc.astype(np.int64))
    _check(d._lib.dsmc_copy_cells(d._h, None, None, None, None))
    d.close()


def test_cells_into_device_memory_on_the_runs_stream():
    """Device arrays are written on the run's own stream and complete on return: a reader on that
    (non-blocking) stream finds them, and work on the default stream is not waited for."""
    import torch

    from paper_2311_14140_gb300 import Dsmc
    from paper_2311_14140_gb300.dsmc import _check
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        d = Dsmc(0.5, N_CELLS, PPC, omega=0.81, body_force=1e-2, seed=3)
        d.step(5)
        want = d.cells()
        t = [torch.zeros(N_CELLS + 1, dtype=torch.int32, device="cuda"),
             torch.zeros(N_CELLS, device="cuda"),
             torch.zeros(N_CELLS, dtype=torch.int64, device="cuda"),
             torch.zeros(N_CELLS, dtype=torch.int64, device="cuda")]
        s.synchronize()
    busy = torch.cuda.Event()
    torch.cuda._sleep(2_000_000_000)  # about a second on the default stream
    busy.record()
    _check(d._lib.dsmc_copy_cells(d._h, *[ctypes.c_void_p(x.data_ptr()) for x in t]))
    with torch.cuda.stream(s):
        got = [x.to("cpu") for x in t]
    waited = busy.query()
    torch.cuda.synchronize()
    for g, w in zip(got, want):
        np.testing.assert_array_equal(g.numpy(), w.astype(g.numpy().dtype))
    assert not waited
    d.close()
