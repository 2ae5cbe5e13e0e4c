"""State kernels above 2^30 particles, where an index plus the number of particles passes 2^31."""
import pytest

pytestmark = pytest.mark.gpu

N_CELLS, PPC = 16384, 65537  # 1,073,758,208 particles: 2^30 + 16,384


def test_state_above_two_to_the_thirty():
    import torch

    from paper_2311_14140_gb300 import Dsmc
    if torch.cuda.mem_get_info()[0] < 90e9:
        pytest.skip("needs 90 GB on the device")
    d = Dsmc(0.5, N_CELLS, PPC, omega=0.5, seed=3)
    got = [torch.full((d.N,), float("nan"), device="cuda") for _ in range(4)]
    d.state_into(*got)
    # drawn cell by cell, PPC to each (the first and the last cells' slots)
    for lo in (0, d.N - 64 * PPC):
        y = got[0][lo:lo + 64 * PPC].double() * N_CELLS
        cell = torch.arange(lo // PPC, lo // PPC + 64, device="cuda").repeat_interleave(PPC)
        # (y in binary32: half a unit of 2^-24 of a position near 1 is 2^-11 of a cell)
        assert (y - cell - 0.5).abs().max().item() <= 0.5 + 2.0 ** -10
    for g in got:
        assert torch.isfinite(g).all().item()
    # a load of the same state, already in cell order, gives it back
    d.load_state(*got, step=0)
    again = [torch.full((d.N,), float("nan"), device="cuda") for _ in range(4)]
    d.state_into(*again)
    for g, a in zip(got, again):
        assert torch.equal(g, a)
    d.close()
    del got, again
    torch.cuda.empty_cache()
