"""Streaming kernel in calls of many rows, on rows on which screening cannot tell the indices apart: equal logits under
T = 0, logits so large that single precision cannot tell their keys apart.  Against the CPU oracle."""
import pytest
import torch

from paper_2504_15475_b200 import workloads as wl

from parity_util import check_sample, check_verify
from test_gpu_unaligned_rows import ersd, guarded, inputs  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [1, 3])
@pytest.mark.parametrize("threads", [128, 256])
@pytest.mark.parametrize("c", [1, 4, 32])
def test_more_ties_than_a_warp_has_room_for(ersd, c, threads, split):  # noqa: F811
    V, B = 7003, 320  # (more rows than the builds for several arrivals take; three tiles of 2048 and a ragged one)
    g = torch.Generator().manual_seed(c)
    z = torch.randn(B, 1, V, generator=g)
    temps = torch.full((B, 1), 0.8)
    z[0::8] = 0.5                             # all alike, greedy: the lowest ids
    temps[0::8] = 0.0
    z[1::8] = 3e7                             # all alike, the screening key's slack is larger than any ln e
    z[2::8] = (z[2::8] * 4).round() / 4       # many ties, greedy
    temps[2::8] = 0.0
    z[3::8, :, 64:] = -3e7                    # a few that may win, the rest far behind
    z[4::8, :, ::3] = float("inf")
    z[5::8, :, 40:] = float("-inf")
    z[6::8] = 3e7
    z[6::8, :, 5000:] = 3.2e7                 # the first chunk's ties are behind the last one's
    seeds = wl.make_seeds(23, c, B)
    tok = torch.full((B, 1, c), -7, dtype=torch.int32, device="cuda")
    ersd.ersd_race_sample(z.cuda(), seeds.cuda(), 1.0, tok, ersd.make_opts(
        top_c=c, kernel_path=1, split_v=split, block_threads=threads, temps=temps.cuda(), temp_strides=(1, 1)))
    torch.cuda.synchronize()
    assert "ersd_race_kernel" in ersd.ersd_last_launch() and "pooled" not in ersd.ersd_last_launch()
    check_sample(z, seeds, 1.0, tok, None, c=c, temps=temps.numpy())


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [5000, 9003])
@pytest.mark.parametrize("parent", [None, [-1, 0, 0, 0, 1, 1]])
@pytest.mark.parametrize("threads", [128, 256])
def test_ties_in_both_rows_of_a_node(ersd, threads, parent, V, dtype):  # noqa: F811
    """Chains, and trees of more than two rows per SM: ties in a node's target row, in its draft row, and in both."""
    B, k = 80, 5
    inp = inputs(B, k, V, "f32", parent=parent)
    inp["T"] = 0.0
    for b in range(0, B, 8):
        for name in ("target", "draft"):
            inp[name][b] = 0.25                                               # both rows of every node
            inp[name][b + 1, :, 3000:] = 9.0
            inp[name][b + 2, :, ::7] = float("inf")
        inp["target"][b + 3] = inp["draft"][b + 4] = -1.5                     # one of them
        inp["draft"][b + 5, :, 2:] = float("-inf")                            # fewer tokens than children
    for name in ("target", "draft"):
        inp[name] = wl._storage(inp[name], dtype)
    on_device = guarded if V % 8 else torch.Tensor.cuda
    out = ersd.verify(on_device(inp["target"]), on_device(inp["draft"]), inp["seeds"].cuda(), 0.0, want_rows=True, parent=parent,
                      kernel_path=1, block_threads=threads)
    torch.cuda.synchronize()
    assert "ersd_race_kernel" in ersd.ersd_last_launch() and "pooled" not in ersd.ersd_last_launch()
    assert check_verify(inp, out) == 0  # (greedy keys are exact: ties go to the lowest id)
