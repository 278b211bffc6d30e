"""Kernels of the library start while the kernel before them on the stream still runs and wait for it
on the device: calls whose inputs the kernels right before them write, with nothing in between, give
the results of calls that are waited for one by one."""
import pytest
import torch

from paper_2504_15475_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ersd():
    from paper_2504_15475_b200 import binding
    binding.lib()
    assert torch.cuda.is_available()
    return binding


@pytest.mark.parametrize("B,k,V,kernel_path", [(1, 4, 20000, 0), (2, 3, 128256, 1), (40, 5, 40001, 0), (3, 2, 3001, 0)])
def test_inputs_written_by_the_previous_kernels(ersd, B, k, V, kernel_path):
    g = torch.Generator(device="cuda").manual_seed(V)
    sets = []
    for n in range(3):
        t = wl.zipf_rows(B * (k + 1), V, g, "cuda").view(B, k + 1, V)
        sets.append(((t).to(torch.bfloat16), (t[:, :k] + 0.7 * torch.randn(B, k, V, generator=g, device="cuda")).to(torch.bfloat16),
                     wl.make_seeds(77, n, B).cuda()))
    tgt, drf, seeds = (torch.empty_like(x) for x in sets[0])
    drafted = torch.empty(B, k, 1, dtype=torch.int32, device="cuda")

    def buffers():
        return [torch.full((B, k + 1), -9, dtype=torch.int32, device="cuda") for _ in range(3)] + \
               [torch.full((B,), -9, dtype=torch.int32, device="cuda") for _ in range(3)]

    def step(n, out, wait):
        def after():
            if wait:
                torch.cuda.synchronize()
        for dst, src in zip((tgt, drf, seeds), sets[n % 3]):
            dst.copy_(src)
        after()
        ersd.ersd_race_sample(drf, seeds, 0.9, drafted, ersd.make_opts(kernel_path=kernel_path))
        after()
        ersd.ersd_verify_tokens(tgt, drafted.view(B, k), seeds, 0.9, out[0], out[3], ersd.make_opts(kernel_path=kernel_path))
        after()
        ersd.ersd_verify(tgt, drf, seeds, 0.9, out[1], out[4], ersd.make_opts(kernel_path=kernel_path))
        after()
        ersd.ersd_gsd_verify(tgt, drf, drafted.view(B, k), seeds, 0.9, out[2], out[5])
        after()

    want = [buffers() for _ in range(3)]
    for n in range(3):
        step(n, want[n], True)
        assert (want[n][0] == want[n][1]).all() and (want[n][3] == want[n][4]).all()
    got = [buffers() for _ in range(30)]
    torch.cuda.synchronize()
    for n in range(30):
        step(n, got[n], False)
    torch.cuda.synchronize()
    for n in range(30):
        assert all((a == b).all() for a, b in zip(got[n], want[n % 3])), n
