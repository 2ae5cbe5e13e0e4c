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
