"""Cluster kernels' short ways: every warp screens a few of its groups of eight indices, and a row whose
contenders all belong to one warp, or to one thread, leaves some of them over; those rows are decided the long
way (one arrival: by every block, with the exact key).  Calls that do not take the short way race the same
rows.  Against the CPU oracle."""
import pytest
import torch

from paper_2504_15475_b200 import workloads as wl

from parity_util import check_sample, check_verify
from test_gpu_unaligned_rows import ersd, guarded, inputs  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def crowd(z, V):
    """Rows 0, 4, ..: contenders in the first warp's groups alone; 1, 5, ..: in one thread's groups of all tiles (tiles
    of 2048 indices that a cluster of 1, 2, 4, 8 or 16 blocks shares out); 2, 6, ..: the row's last group; 3, 7, ..: as drawn."""
    flat = z.view(-1, V)
    flat[0::4, :min(V, 256)] += 9.0
    for i in range(0, V, 2048):
        flat[1::4, i + 16:i + 24] += 9.0
    flat[2::4, (V - 1) // 8 * 8:] += 9.0


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("B,V", [(40, 700), (40, 2048), (20, 4100), (10, 16384), (6, 32001), (2, 66000), (1, 131080),
                                 (2, 66001), (6, 33001), (4, 50001)])
def test_contenders_of_one_warp_and_of_one_thread(ersd, B, V, dtype):  # noqa: F811
    """Clusters of one or two blocks (the long way), of four, eight and sixteen."""
    k, short = 3, V > 16384
    inp = inputs(B, k, V, "f32")
    for name in ("target", "draft"):
        crowd(inp[name], V)
        inp[name] = wl._storage(inp[name], dtype)
    on_device = guarded if V % 8 else torch.Tensor.cuda
    seeds = inp["seeds"].cuda()
    for T in (0.8, 3.0, 0.0):
        inp["T"] = T
        out = ersd.verify(on_device(inp["target"]), on_device(inp["draft"]), seeds, T, want_rows=True)
        torch.cuda.synchronize()
        assert "ersd_cluster_kernel" in ersd.ersd_last_launch() and "(unstaged)" not in ersd.ersd_last_launch()
        assert ("short way" in ersd.ersd_last_launch()) == short
        check_verify(inp, out)
        tok = torch.full((B, k + 1, 1), -7, dtype=torch.int32, device="cuda")
        key = torch.full((B, k + 1, 1), -7.0, dtype=torch.float32, device="cuda")
        ersd.ersd_race_sample(on_device(inp["target"]), seeds, T, tok, ersd.make_opts(out_key=key))
        torch.cuda.synchronize()
        assert "(unstaged)" not in ersd.ersd_last_launch() and ("short way" in ersd.ersd_last_launch()) == short
        check_sample(inp["target"], inp["seeds"], T, tok, key)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("B,V,c", [(4, 131072, 2), (2, 100001, 4), (1, 131080, 8), (4, 128256, 12), (1, 40961, 5), (40, 70001, 4),
                                   (30, 128256, 3), (30, 100001, 2), (36, 133000, 2)])
def test_several_arrivals_of_one_warp_and_of_one_thread(ersd, B, V, c, dtype):  # noqa: F811
    """Staged and not; rows of ties, rows with fewer tokens than arrivals, infinities, and rows as drawn."""
    inp = inputs(2 * B, 0, V, "f32")
    z = inp["target"]
    crowd(z, V)
    flat = z.view(-1, V)
    if B > 1:
        flat[B] = 0.5                        # under T = 0 a tie of the whole row
        flat[B + 1, 3:] = float("-inf")      # three tokens
    if B > 3:
        flat[B + 2, V - 1] = float("inf")
        flat[B + 3] = (flat[B + 3] * 2).round() / 2
    z = wl._storage(z, dtype)
    on_device = guarded if V % 8 else torch.Tensor.cuda
    for T in (0.8, 2.5, 0.0):
        tok = torch.full((2 * B, 1, c), -7, dtype=torch.int32, device="cuda")
        key = torch.full((2 * B, 1, c), -7.0, dtype=torch.float32, device="cuda")
        ersd.ersd_race_sample(on_device(z), inp["seeds"].cuda(), T, tok, ersd.make_opts(top_c=c, out_key=key))
        torch.cuda.synchronize()
        assert "ersd_cluster_top_kernel" in ersd.ersd_last_launch()
        # (80 rows get clusters of 32 warps: too few for four arrivals; greedy calls go the long way)
        assert ("short way" in ersd.ersd_last_launch()) == (B < 40 and T > 0)
        check_sample(z, inp["seeds"], T, tok, key, c=c)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [900, 40000, 128256])
def test_key_of_a_greedy_row_of_zeros(ersd, V, dtype):  # noqa: F811
    """-z, without a sign, whether the row goes the short way or, all groups being tied, the long one."""
    z = torch.zeros(2, 1, V, dtype=dtype, device="cuda")
    z[1, 0, 5:] = -1.0
    tok = torch.full((2, 1, 1), -7, dtype=torch.int32, device="cuda")
    key = torch.full((2, 1, 1), -7.0, dtype=torch.float32, device="cuda")
    ersd.ersd_race_sample(z, wl.make_seeds(3, 0, 2).cuda(), 0.0, tok, ersd.make_opts(out_key=key))
    torch.cuda.synchronize()
    assert "ersd_cluster_kernel" in ersd.ersd_last_launch()
    assert (tok == 0).all() and (key.view(torch.int32) == 0).all()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_greedy_rows_among_others(ersd, dtype):  # noqa: F811
    """A call whose rows have temperatures of their own takes the short way's build, in which greedy rows go the long way."""
    B, V, c = 12, 100008, 4
    z = inputs(B, 0, V, "f32")["target"]
    crowd(z, V)
    z[8:] = (z[8:] * 2).round() / 2
    temps = torch.tensor([0.8, 0.0]).repeat(B // 2).view(B, 1).contiguous()
    z, seeds = wl._storage(z, dtype), wl.make_seeds(31, c, B)
    tok = torch.full((B, 1, c), -7, dtype=torch.int32, device="cuda")
    key = torch.full((B, 1, c), -7.0, dtype=torch.float32, device="cuda")
    ersd.ersd_race_sample(z.cuda(), seeds.cuda(), 1.0, tok, ersd.make_opts(top_c=c, out_key=key, temps=temps.cuda(), temp_strides=(1, 1)))
    torch.cuda.synchronize()
    assert "ersd_cluster_top_kernel" in ersd.ersd_last_launch() and "short way" in ersd.ersd_last_launch()
    check_sample(z, seeds, 1.0, tok, key, c=c, temps=temps.numpy())


@pytest.mark.parametrize("name", ["specinfer", "4x4"])
def test_trees_whose_rows_have_a_cluster_each(ersd, name):  # noqa: F811
    parent = {"specinfer": wl.TREE_SPECINFER, "4x4": wl.TREE_4x4}[name]
    for V, T in ((128256, 0.8), (70001, 3.0), (40000, 0.0)):
        inp = inputs(1, len(parent) - 1, V, "f32", parent=parent)
        inp["T"] = T
        for n in ("target", "draft"):
            crowd(inp[n], V)
            inp[n] = wl._storage(inp[n], "bf16")
        on_device = guarded if V % 8 else torch.Tensor.cuda
        out = ersd.verify(on_device(inp["target"]), on_device(inp["draft"]), inp["seeds"].cuda(), T, want_rows=True, parent=list(parent))
        torch.cuda.synchronize()
        assert "ersd_cluster_top_kernel" in ersd.ersd_last_launch()
        assert "1 row(s) per cluster" in ersd.ersd_last_launch() and ("short way" in ersd.ersd_last_launch()) == (T > 0)
        check_verify(inp, out)
