"""Cluster kernel over rows that are not staged in shared memory (calls of more than a few megabytes of
logits): against the CPU oracle at the edges of its tiles, clusters and block sizes, and against the
streaming kernel on special values."""
import pytest
import torch

from paper_2504_15475_b200 import workloads as wl

from parity_util import check_sample, check_verify
from test_gpu_unaligned_rows import ersd, guarded, inputs  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# positions x vocabulary: blocks of 128 threads by themselves, of 256 by themselves, in clusters of 2, 4, 8, 16
# whose last tile is ragged, ends on a tile's edge, or leaves blocks with one tile less
SHAPES = [(1300, 2047), (1300, 2048), (2400, 1026), (600, 16384), (600, 16385), (150, 32001), (150, 24576), (60, 40961),
          (40, 66001), (20, 131080), (18, 139166)]


def unstaged(ersd):
    assert "ersd_cluster_kernel" in ersd.ersd_last_launch() and "(unstaged)" in ersd.ersd_last_launch()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("positions,V", SHAPES)
def test_against_the_oracle(ersd, positions, V, dtype):  # noqa: F811
    k = 1
    inp = inputs(positions // 2, k, V, dtype)
    on_device = guarded if V % 8 else torch.Tensor.cuda
    out = ersd.verify(on_device(inp["target"]), on_device(inp["draft"]), inp["seeds"].cuda(), inp["T"], want_rows=True)
    torch.cuda.synchronize()
    unstaged(ersd)
    check_verify(inp, out)
    if positions * V * (2 if dtype == "bf16" else 4) > 8 << 20:
        logits, seeds = inp["target"], inp["seeds"]
        B = positions // 2
        tok = torch.full((B, k + 1, 1), -7, dtype=torch.int32, device="cuda")
        key = torch.full((B, k + 1, 1), -7.0, dtype=torch.float32, device="cuda")
        ersd.ersd_race_sample(on_device(logits), seeds.cuda(), 0.8, tok, ersd.make_opts(out_key=key))
        torch.cuda.synchronize()
        unstaged(ersd)
        check_sample(logits, seeds, 0.8, tok, key)


@pytest.mark.parametrize("positions,V", [(20, 128256), (100, 128256), (96, 40960), (48, 65544), (112, 24584)])
def test_three_tiles_ahead(ersd, positions, V):  # noqa: F811
    """Aligned pairs of bf16 rows, up to three blocks to an SM: 5 to 16 tiles to a block, whole and ragged."""
    inp = inputs(positions // 2, 1, V, "bf16")
    out = ersd.verify(inp["target"].cuda(), inp["draft"].cuda(), inp["seeds"].cuda(), inp["T"], want_rows=True)
    torch.cuda.synchronize()
    unstaged(ersd)
    assert "more tiles ahead" in ersd.ersd_last_launch(), ersd.ersd_last_launch()
    check_verify(inp, out)


@pytest.mark.parametrize("rows,V,more", [(100, 32000, False), (450, 34816, True), (450, 34817, True), (450, 32768, True), (450, 30720, False), (300, 38912, False),
                                         (150, 151936, True), (230, 69640, True)])
def test_32_bit_rows_two_tiles_ahead(ersd, rows, V, more):  # noqa: F811
    """One row per position: 16 tiles to a block and more, in more than three blocks to an SM."""
    logits = inputs(rows, 0, V, "f32")["target"]
    seeds = wl.make_seeds(7, V, rows)
    tok = torch.full((rows, 1, 1), -7, dtype=torch.int32, device="cuda")
    key = torch.full((rows, 1, 1), -7.0, dtype=torch.float32, device="cuda")
    on_device = guarded if V % 8 else torch.Tensor.cuda
    ersd.ersd_race_sample(on_device(logits), seeds.cuda(), 0.8, tok, ersd.make_opts(out_key=key))
    torch.cuda.synchronize()
    unstaged(ersd)
    assert ("more tiles ahead" in ersd.ersd_last_launch()) == more, ersd.ersd_last_launch()
    check_sample(logits, seeds, 0.8, tok, key)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_special_values_as_in_the_streaming_kernel(ersd, dtype):  # noqa: F811
    V, B = 5000, 160
    g = torch.Generator().manual_seed(9)
    t = torch.randn(B, 4, V, generator=g)
    d = t[:, :3] + 0.1 * torch.randn(B, 3, V, generator=g)
    t[0::8, 0, :] = float("-inf")                     # fully masked rows
    t[1::8, 0, 5] = float("nan")
    t[1::8, 0, 100:] = float("-inf")
    d[1::8, 0, 4017] = float("inf")                   # +inf always wins
    d[2::8, 0, :] = float("nan")
    t[3::8, 1, :] = float("inf")                      # every key the smallest there is
    t[4::8, 2, :] = 0.25                              # all alike: with T = 0 a tie of the whole row
    d[5::8, 1, 1:] = d[5::8, 1, 0:1]
    temps = torch.full((B, 4), 0.7)
    temps[6::8, 1] = -1.0                             # not a temperature: no arrivals
    temps[7::8, 2] = 0.0
    t, d, seeds = wl._storage(t, dtype).cuda(), wl._storage(d, dtype).cuda(), wl.make_seeds(3, 0, B).cuda()
    for T, tt in ((0.8, None), (0.0, None), (1.0, temps)):
        kw = {} if tt is None else dict(temps=tt.cuda())
        a = ersd.verify(t, d, seeds, T, want_rows=True, kernel_path=2, **kw)
        unstaged(ersd)
        b = ersd.verify(t, d, seeds, T, want_rows=True, kernel_path=1, **kw)
        torch.cuda.synchronize()
        for name in a:
            assert torch.equal(a[name], b[name]) or (name.endswith("key") and (a[name] == b[name]).all()), (name, T)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("B,V", [(160, 2049), (24, 16384), (10, 32001), (6, 66001), (3, 131080)])
def test_several_arrivals_against_the_oracle(ersd, B, V, dtype):  # noqa: F811
    """Blocks by themselves and clusters of 2 to 16, ragged last tiles, rows on and off 16-byte boundaries."""
    on_device = guarded if V % 8 else torch.Tensor.cuda
    parent = wl.TREE_SPECINFER
    inp = inputs(B, len(parent) - 1, V, dtype, parent=parent)
    out = ersd.verify(on_device(inp["target"]), on_device(inp["draft"]), inp["seeds"].cuda(), inp["T"], want_rows=True,
                      parent=list(parent))
    torch.cuda.synchronize()
    assert "ersd_cluster_top_kernel" in ersd.ersd_last_launch() and "(unstaged)" in ersd.ersd_last_launch()
    check_verify(inp, out)
    logits, seeds, c = inp["target"], inp["seeds"], 32
    tok = torch.full((B, len(parent), c), -7, dtype=torch.int32, device="cuda")
    key = torch.full((B, len(parent), c), -7.0, dtype=torch.float32, device="cuda")
    ersd.ersd_race_sample(on_device(logits), seeds.cuda(), 0.8, tok, ersd.make_opts(top_c=c, out_key=key))
    torch.cuda.synchronize()
    assert "ersd_cluster_top_kernel" in ersd.ersd_last_launch() and "(unstaged)" in ersd.ersd_last_launch()
    check_sample(logits, seeds, 0.8, tok, key, c=c)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_several_arrivals_of_tied_and_masked_rows(ersd, dtype):  # noqa: F811
    """Rows of equal logits under T = 0 overflow a block's lists; rows with fewer tokens than arrivals wanted."""
    V, B, c = 40008, 60, 8
    g = torch.Generator().manual_seed(19)
    z = torch.randn(B, 1, V, generator=g)
    z[0::5] = 0.5
    z[1::5, :, 3:] = float("-inf")
    z[2::5, :, ::2] = float("nan")
    z[3::5, :, 17] = float("inf")
    temps = torch.full((B, 1), 0.9)
    temps[0::2] = 0.0
    temps[7] = float("nan")
    z, seeds = wl._storage(z, dtype).cuda(), wl.make_seeds(5, 0, B).cuda()
    got = []
    for path in (2, 1):
        tok = torch.full((B, 1, c), -7, dtype=torch.int32, device="cuda")
        key = torch.full((B, 1, c), -7.0, dtype=torch.float32, device="cuda")
        ersd.ersd_race_sample(z, seeds, 1.0, tok, ersd.make_opts(top_c=c, out_key=key, kernel_path=path, temps=temps.cuda(),
                                                                 temp_strides=(1, 1)))
        torch.cuda.synchronize()
        assert ("(unstaged)" in ersd.ersd_last_launch()) == (path == 2)
        got.append((tok, key))
    assert torch.equal(got[0][0], got[1][0])
    assert (got[0][1] == got[1][1]).all()
