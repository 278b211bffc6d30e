"""A call that fails leaves nothing behind: neither an error that the next call on the thread, or another
library's launch check, would take for its own, nor anything in the scratch memory."""
import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ersd():
    from paper_2504_15475_b200 import binding
    binding.lib()
    assert torch.cuda.is_available()
    return binding


def test_a_failed_call_leaves_no_error_to_the_next(ersd):
    L = ersd.lib()
    row = torch.zeros(64, dtype=torch.bfloat16, device="cuda")
    seeds = torch.zeros(64, dtype=torch.int64, device="cuda")
    out = torch.empty(64, dtype=torch.float32, device="cuda")
    ptr = [C.c_void_p(t.data_ptr()) for t in (row, seeds, out)]
    # a private workspace of some terabytes: the allocation is refused before anything is launched
    assert L.ersd_verify(ptr[0], ptr[0], 1, ptr[1], 8000000, 255, 1, 1.0, ptr[2], ptr[2], None, None) == -4
    assert L.ersd_last_cuda_error() == 2   # cudaErrorMemoryAllocation
    assert L.ersd_row_keys(ptr[0], 1, 64, 1.0, 1, 0, 0, 0, ptr[2], None) == 0
    torch.cuda.synchronize()
    assert torch.isfinite(out).all()
