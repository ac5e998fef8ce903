"""A wait that cannot succeed ends by the clock, however many polls it is allowed."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_wait_ends_by_the_clock(zipvl):
    """2^20 polls take four seconds; the wait gives up after one and a half, and reports it."""
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    progress = torch.full((4,), -1, dtype=torch.int32, device=DEV)
    zipvl.zipvl_selftest_wait_timeout(16, progress, st)                 # (loads the kernel)
    st.zero_()
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    a.record()
    zipvl.zipvl_selftest_wait_timeout(1 << 20, progress, st)
    b.record()
    torch.cuda.synchronize()
    assert st.item() == zipvl.DEV_TIMEOUT and progress.tolist() == [1, 0, 0, 0]
    assert 1400 < a.elapsed_time(b) < 2000
