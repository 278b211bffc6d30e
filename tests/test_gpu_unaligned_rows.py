"""Logit rows that start on no 16-byte boundary (a vocabulary that is no multiple of eight): every
kernel against the CPU oracle, through the C boundary.  The tensors sit between guard elements that
must never be raced, one element off a boundary themselves."""
import pytest
import torch

from paper_2504_15475_b200 import workloads as wl

from parity_util import check_sample, check_verify

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ersd():
    from paper_2504_15475_b200 import binding
    binding.lib()
    assert torch.cuda.is_available()
    return binding


def guarded(t):
    """A copy of t on the device, one element off a 16-byte boundary, between logits that always win."""
    flat = torch.full((t.numel() + 24,), float("inf"), dtype=t.dtype, device="cuda")
    flat[9:9 + t.numel()] = t.reshape(-1).cuda()
    return flat[9:9 + t.numel()].view(t.shape)


def inputs(B, k, V, dtype, parent=None, T=0.8):
    w = wl.Workload("unaligned", B=B, k=k, V=V, dtype=dtype, sigma=0.7, T=T, config_id=90 + V % 7, parent=parent)
    return wl.make_inputs(w)


def run(ersd, inp, **kw):
    parent = inp["parent"]
    out = ersd.verify(guarded(inp["target"]), guarded(inp["draft"]), inp["seeds"].cuda(), inp["T"],
                      parent=None if parent is None else list(parent), want_rows=True, **kw)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [1, 3, 9, 15, 2047, 2049, 4091, 32001, 50003])
def test_few_rows(ersd, V, dtype):
    """Cluster kernel: ragged ends, tiles that end within a 16-byte unit of the row's end."""
    inp = inputs(2, 3, V, dtype)
    out = run(ersd, inp)
    assert "ersd_cluster_kernel" in ersd.ersd_last_launch()
    check_verify(inp, out)
    logits, seeds = inp["target"], inp["seeds"]
    tok = torch.full((2, 4, 1), -7, dtype=torch.int32, device="cuda")
    key = torch.full((2, 4, 1), -7.0, dtype=torch.float32, device="cuda")
    ersd.ersd_race_sample(guarded(logits), seeds.cuda(), 0.8, tok, ersd.make_opts(out_key=key))
    torch.cuda.synchronize()
    assert "ersd_cluster_kernel" in ersd.ersd_last_launch()
    check_sample(logits, seeds, 0.8, tok, key)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [9, 2049, 20003])
def test_few_rows_of_several_arrivals(ersd, V, dtype):
    inp = inputs(2, len(wl.TREE_SPECINFER) - 1, V, dtype, parent=wl.TREE_SPECINFER)
    out = run(ersd, inp)
    assert "ersd_cluster_top_kernel" in ersd.ersd_last_launch()
    check_verify(inp, out)
    c = min(8, V)
    logits, seeds = inp["target"][:, :3].contiguous(), inp["seeds"]
    tok = torch.full((2, 3, c), -7, dtype=torch.int32, device="cuda")
    key = torch.full((2, 3, c), -7.0, dtype=torch.float32, device="cuda")
    ersd.ersd_race_sample(guarded(logits), seeds.cuda(), 0.9, tok, ersd.make_opts(top_c=c, out_key=key))
    torch.cuda.synchronize()
    assert "ersd_cluster_top_kernel" in ersd.ersd_last_launch()
    check_sample(logits, seeds, 0.9, tok, key, c=c)


@pytest.mark.parametrize("V", [5, 1024, 1030, 3001])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_many_short_rows_take_small_blocks(ersd, V, dtype):
    """More positions than 256-thread blocks are resident: one block of 128 threads per position."""
    inp = inputs(150, 4, V, dtype)
    out = run(ersd, inp)
    assert "x 128 threads" in ersd.ersd_last_launch()
    check_verify(inp, out)
    logits, seeds = inp["target"], inp["seeds"]
    tok = torch.full((150, 5, 1), -7, dtype=torch.int32, device="cuda")
    key = torch.full((150, 5, 1), -7.0, dtype=torch.float32, device="cuda")
    ersd.ersd_race_sample(logits.cuda(), seeds.cuda(), 0.8, tok, ersd.make_opts(out_key=key))
    torch.cuda.synchronize()
    assert "x 128 threads" in ersd.ersd_last_launch()
    check_sample(logits, seeds, 0.8, tok, key)


@pytest.mark.parametrize("threads", [128, 256])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [3, 1027, 2055, 4097, 8199, 16390, 40001])
def test_streaming_kernel(ersd, V, dtype, threads):
    """The ring over memory's 16-byte units: chunks of few tiles, two ragged tiles at a row's end, every shift."""
    inp = inputs(4, 3, V, dtype)
    for split in (0, 3):
        out = run(ersd, inp, kernel_path=1, block_threads=threads, split_v=split)
        assert "ersd_race_kernel" in ersd.ersd_last_launch()
        check_verify(inp, out)
    tree = inputs(2, len(wl.TREE_4x4) - 1, V, dtype, parent=wl.TREE_4x4)
    out = run(ersd, tree, kernel_path=1, block_threads=threads)
    assert "ersd_race_kernel" in ersd.ersd_last_launch()
    check_verify(tree, out)
