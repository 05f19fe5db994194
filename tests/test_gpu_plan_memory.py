"""A destroyed plan gives back all of its device memory."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


@pytest.mark.parametrize("fft", ["auto", "cufft"])
def test_plans_leave_no_memory_behind(gb, fft):
    def make():
        gb.Plan(np.eye(3) * 30.0, (32, 32, 33), 4, 0.3, 9.0, max_ions=1 << 18, fft=fft, brick=(8, 8, 16)).close()
        torch.cuda.synchronize()

    make()   # what the library itself keeps
    make()
    before = torch.cuda.mem_get_info()[0]
    for _ in range(16):
        make()
    # 16 plans of 2^18 ions: any per-ion array of 16 bytes left behind is 64 MiB
    assert before - torch.cuda.mem_get_info()[0] < 32 << 20
