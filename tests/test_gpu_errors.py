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


def test_more_sequences_than_the_launch_grid_takes(ersd):
    """Refused on the host, before the first of the call's two kernels is on the stream."""
    B = 65536
    tgt = torch.zeros(B, 1, 8, dtype=torch.bfloat16, device="cuda")
    seeds = torch.arange(B, device="cuda")
    out = torch.full((B, 1), -9, dtype=torch.int32, device="cuda")
    acc = torch.full((B,), -9, dtype=torch.int32, device="cuda")
    ws = torch.zeros(ersd.ersd_workspace_bytes(B, 1), dtype=torch.uint8, device="cuda")
    with pytest.raises(ersd.ErsdError) as e:
        ersd.ersd_gsd_verify(tgt, None, None, seeds, 1.0, out, acc, ersd.make_opts(workspace=ws))
    assert e.value.status == -3
    torch.cuda.synchronize()
    assert (ws == 0).all() and (out == -9).all()
    ersd.ersd_gsd_verify_tree(tgt[:4].contiguous(), None, None, [-1], seeds[:4].contiguous(), 1.0, out, acc)
    ersd.ersd_gsd_verify(tgt[:65535].contiguous(), None, None, seeds[:65535].contiguous(), 1.0, out, acc,
                         ersd.make_opts(workspace=ws))
    torch.cuda.synchronize()
    assert (acc[:65535] == 0).all() and (out[:65535] >= 0).all() and (out[:65535] < 8).all()
