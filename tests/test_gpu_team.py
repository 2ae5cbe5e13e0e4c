"""Teams of CTAs over the device (runs of 40,000 to about 1.3 million particles)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ERR_TEAM = 256  # the error word's bit for a wait between the CTAs of a team that ran out


def _snapshot(d):
    m, n = d.moments()
    return (*d.state(), *d.cells(), m, np.int64(n))


def _assert_same(a, b):
    for k, (x, y) in enumerate(zip(a, b)):
        x, y = np.ascontiguousarray(x), np.ascontiguousarray(y)
        np.testing.assert_array_equal(x.view(np.uint8), y.view(np.uint8), err_msg=f"output {k}")


def test_steps_behind_a_lost_team_leave_the_run_alone():
    """Once a wait has run out, the barrier's counter is out of step.  Launches that were queued
    behind it must not start: the run keeps the state it has, and the call that synchronises
    reports the error.  The error word (the first of the workspace's last 256 bytes) is set here
    by hand."""
    import torch

    from paper_2311_14140_gb300 import Dsmc, DsmcError
    d = Dsmc(0.3, 400, 103, omega=0.81, body_force=1e-3, seed=2)
    d.step(6)
    assert d.last_step()[0] == "team"
    before = _snapshot(d)
    word = d._ws[d.info()["device_bytes"] - 256:][:4].view(torch.int32)
    assert word.item() == 0
    word.fill_(ERR_TEAM)
    d.step(4)  # (even: the same buffers hold the state afterwards)
    d.step(2)
    with pytest.raises(DsmcError, match="team-barrier-timeout"):
        d.sync()
    with pytest.raises(DsmcError):
        d.step(1)  # latched
    word.fill_(0)
    after = _snapshot(d)
    d.close()
    _assert_same(before[:-1], after[:-1])  # (but for the host's count of sampled steps)


def test_runs_on_several_streams():
    """Two runs in flight keep their teams; a third one's steps overlap with them as span passes,
    and on its own again it is a team.  All evolve as alone.  (A second's wait at the head of each
    stream keeps the steps in flight.)"""
    import torch

    from paper_2311_14140_gb300 import Dsmc
    sizes = [(400, 103), (200, 500), (37, 2000)]
    want, runs, streams = [], [], []
    for k, (n_cells, ppc) in enumerate(sizes):
        args = dict(omega=0.81, body_force=1e-3, seed=k)
        with Dsmc(0.3, n_cells, ppc, **args) as d:
            for _ in range(3):
                d.step(5)
            assert d.last_step()[0] == "team"
            want.append(_snapshot(d))
        streams.append(torch.cuda.Stream())
        with torch.cuda.stream(streams[k]):
            runs.append(Dsmc(0.3, n_cells, ppc, **args))
    for d in runs:  # one after the other: each has the device to itself
        d.step(5)
        assert d.last_step()[0] == "team"
        d.sync()
    kinds = []
    for d, s in zip(runs, streams):
        with torch.cuda.stream(s):
            torch.cuda._sleep(2_000_000_000)
        d.step(5)
        kinds.append(d.last_step()[0])
    assert kinds == ["team", "team", "spans"]
    for d in runs:
        d.sync()
    runs[2].step(5)
    assert runs[2].last_step()[0] == "team"
    runs[0].step(5)
    runs[1].step(5)
    for d, w in zip(runs, want):
        _assert_same(_snapshot(d), w)
    for d in runs:
        d.close()


def test_runs_of_several_threads():
    """Six runs stepped by a thread each, on their own streams, created and closed while others
    step: whichever way each call's steps take, every run evolves as alone."""
    import threading

    import torch

    from paper_2311_14140_gb300 import Dsmc
    sizes = [(400, 103), (200, 500), (37, 2000), (500, 400), (1200, 50), (20, 30000)]

    def evolve(k, stream):
        with torch.cuda.stream(stream):
            d = Dsmc(0.3, *sizes[k], omega=0.5, body_force=1e-3, seed=k)
            for n in (1, 7, 2, 30, 5, 40, 3):
                d.step(n)
            out = _snapshot(d)
            d.close()
        return out

    want = [evolve(k, torch.cuda.current_stream()) for k in range(len(sizes))]
    got, errors = [[] for _ in sizes], []

    def work(k):
        try:
            for _ in range(4):
                got[k].append(evolve(k, torch.cuda.Stream()))
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for g, w in zip(got, want):
        for x in g:
            _assert_same(x, w)


def test_steps_while_another_stream_is_captured():
    """A capture of another stream in global mode, which forbids event queries, is not disturbed by
    the steps of three runs on teams in another thread."""
    import threading

    import torch

    from paper_2311_14140_gb300 import Dsmc
    runs = []
    for k in range(3):
        with torch.cuda.stream(torch.cuda.Stream()):
            d = Dsmc(0.3, 200, 300, omega=0.5, body_force=1e-3, seed=k)
            d.step(2)
            d.sync()
            runs.append(d)
    x = torch.zeros(1024, device="cuda")
    torch.cuda.synchronize()
    errors = []

    def work():
        try:
            for d in runs:
                d.step(8)
        except Exception as e:  # reported by the main thread
            errors.append(e)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        x += 1.0
        t = threading.Thread(target=work)
        t.start()
        t.join()
    g.replay()
    torch.cuda.synchronize()
    assert not errors
    assert x.min().item() == 1.0
    for d in runs:
        assert d.info()["step"] == 10
        d.sync()
        d.close()
