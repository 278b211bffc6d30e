"""Greedy speculative decoding on the GPU (ersd_gsd_verify, ersd_gsd_verify_tree) against the CPU
oracle's Algorithms 1 and 4, through the C boundary, on the same seeded inputs.

Bar: emitted tokens and accept lengths equal the oracle's.  Both sides decide in double precision,
so the allowed exceptions are decisions within rounding of each other, which the oracle's outputs
expose: a ratio test with |ratio - u| < 1e-9 * ratio, or a final race whose two best arrival times
are closer than 1e-5 relative (the near-tie window); such sequences are counted."""
import numpy as np
import pytest
import torch

import oracle
from paper_2504_15475_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ersd():
    from paper_2504_15475_b200 import binding
    binding.lib()
    assert torch.cuda.is_available()
    return binding


def draft_tokens(ersd, draft, seeds, T, c=1, temps=None):
    """Tokens drafted on the GPU: the first c arrivals of every draft row's race (a sample without
    replacement of that row's law)."""
    B, R, V = draft.shape
    tok = torch.empty(B, R, c, dtype=torch.int32, device="cuda")
    kw = {}
    if temps is not None:
        kw = dict(temps=temps, temp_strides=(temps.stride(0), temps.stride(1)))
    ersd.ersd_race_sample(draft, seeds, T, tok, ersd.make_opts(top_c=c, **kw))
    return tok


def ambiguous(ref):
    """Sequences whose outcome hangs on a decision within rounding (see the module docstring)."""
    amb = np.zeros(ref["accept_len"].shape[0], bool)
    if "ratio" in ref:
        r, u = ref["ratio"], ref["unif"]
        with np.errstate(invalid="ignore"):
            amb |= (np.abs(r - u) < 1e-9 * np.maximum(r, 1e-300)).any(axis=1)
    t = ref["last_times"]
    with np.errstate(invalid="ignore"):
        amb |= (t[:, 1] - t[:, 0]) < 1e-5 * t[:, 0]
    return amb


@pytest.mark.parametrize("name,scale", [("c1", {}), ("c2", {}), ("c5", dict(B=12)), ("c3", dict(B=4)),
                                        ("c2", dict(B=300, V=3000))])
def test_sequence_gsd_against_the_oracle(ersd, name, scale):
    w = wl.scaled(wl.CONFIGS[name], **scale)
    inp = wl.make_inputs(w, call=5)
    tgt, drf, seeds = inp["target"].cuda(), inp["draft"].cuda(), inp["seeds"].cuda()
    temps = None if inp.get("temps") is None else inp["temps"].cuda()
    kw = {} if temps is None else dict(temps=temps, temp_strides=(temps.stride(0), temps.stride(1)))
    t_d = None if temps is None else temps[:, :w.k].contiguous()
    tok = draft_tokens(ersd, drf, seeds, inp["T"], temps=t_d)[..., 0].contiguous()
    out = torch.full((w.B, w.k + 1), -9, dtype=torch.int32, device="cuda")
    acc = torch.full((w.B,), -9, dtype=torch.int32, device="cuda")
    for rep in range(2):                        # twice: the call leaves the workspace as it found it
        ersd.ersd_gsd_verify(tgt, drf, tok, seeds, inp["T"], out, acc, ersd.make_opts(**kw))
    torch.cuda.synchronize()
    ref = oracle.gsd_verify(wl.as_numpy_logits(inp["target"]), wl.as_numpy_logits(inp["draft"]),
                            tok.cpu().numpy(), wl.seeds_as_u64(inp["seeds"]), T=inp["T"],
                            temps=None if temps is None else inp["temps"].numpy())
    amb = ambiguous(ref)
    assert amb.sum() <= 1
    ok = ~amb
    assert (acc.cpu().numpy()[ok] == ref["accept_len"][ok]).all()
    assert (out.cpu().numpy()[ok] == ref["tokens"][ok]).all()
    assert 0 < ref["accept_len"].mean() < w.k or w.B == 1   # both outcomes occur
    # an ERSD call afterwards finds its workspace in order
    from parity_util import check_verify
    res = ersd.verify(tgt, drf, seeds, inp["T"], temps=temps, want_rows=True)
    torch.cuda.synchronize()
    check_verify(inp, res)


def test_sequence_gsd_options_and_errors(ersd):
    w = wl.scaled(wl.CONFIGS["c2"], B=5, V=5000)
    inp = wl.make_inputs(w, call=9)
    tgt, drf, seeds = inp["target"].cuda(), inp["draft"].cuda(), inp["seeds"].cuda()
    seq = torch.tensor([7, 7, 9, 11, 12], dtype=torch.int32, device="cuda")
    off = torch.tensor([0, 5, 100, 3, 0], dtype=torch.int32, device="cuda")
    tok = torch.randint(0, w.V, (w.B, w.k), dtype=torch.int32, device="cuda")   # any tokens may be verified
    ws = torch.empty(ersd.ersd_workspace_bytes(w.B, w.k + 1), dtype=torch.uint8, device="cuda")
    ersd.ersd_workspace_init(ws)
    out = torch.empty(w.B, w.k + 1, dtype=torch.int32, device="cuda")
    acc = torch.empty(w.B, dtype=torch.int32, device="cuda")
    ersd.ersd_gsd_verify(tgt, drf, tok, seeds, 0.8, out, acc, ersd.make_opts(seq_ids=seq, pos_offsets=off, workspace=ws))
    torch.cuda.synchronize()
    assert (ws == 0).all()                                       # left zeroed
    ref = oracle.gsd_verify(wl.as_numpy_logits(inp["target"]), wl.as_numpy_logits(inp["draft"]), tok.cpu().numpy(),
                            wl.seeds_as_u64(inp["seeds"]), T=0.8, seq_ids=seq.cpu().numpy(), pos_offsets=off.cpu().numpy())
    assert not ambiguous(ref).any()
    assert (acc.cpu().numpy() == ref["accept_len"]).all() and (out.cpu().numpy() == ref["tokens"]).all()
    for bad_T in (0.0, -1.0, float("nan")):
        with pytest.raises(ersd.ErsdError) as e:
            ersd.ersd_gsd_verify(tgt, drf, tok, seeds, bad_T, out, acc)
        assert e.value.status == -1
    with pytest.raises(ersd.ErsdError) as e:
        ersd.ersd_gsd_verify(tgt, drf, None, seeds, 1.0, out, acc)
    assert e.value.status == -1
    # no drafts: one sample of the only target row
    ersd.ersd_gsd_verify(tgt[:, :1].contiguous(), None, None, seeds, 1.0, out[:, :1].contiguous(), acc)
    torch.cuda.synchronize()
    assert (acc == 0).all()


@pytest.mark.parametrize("parent,B,V", [(wl.TREE_4x4, 6, 20000), (wl.TREE_SPECINFER, 4, 151936), (wl.star_parent(5), 8, 4097),
                                         (wl.chain_parent(4), 5, 32000), ([-1], 3, 1000)])
def test_tree_gsd_against_the_oracle(ersd, parent, B, V):
    nodes = len(parent)
    w = wl.Workload("gsdtree", B=B, k=nodes - 1, V=V, dtype="bf16", sigma=0.7, T=1.0, config_id=50, parent=tuple(parent))
    inp = wl.make_inputs(w, call=2)
    tgt, drf, seeds = inp["target"].cuda(), inp["draft"].cuda(), inp["seeds"].cuda()
    _, max_c, nchild, rank = oracle.tree_shape(parent)
    arr = draft_tokens(ersd, drf, seeds, inp["T"], c=max_c)      # [B, nodes, max_c]: arrivals of every node's draft race
    tok = torch.full((B, nodes), -1, dtype=torch.int32, device="cuda")
    for n in range(1, nodes):
        tok[:, n] = arr[:, parent[n], rank[n]]
    D = ersd.ersd_tree_depth(parent)
    out = torch.full((B, D + 1), -9, dtype=torch.int32, device="cuda")
    acc = torch.full((B,), -9, dtype=torch.int32, device="cuda")
    path = torch.full((B, D + 1), -9, dtype=torch.int32, device="cuda")
    ersd.ersd_gsd_verify_tree(tgt, drf, tok, parent, seeds, inp["T"], out, acc, ersd.make_opts(out_path=path))
    torch.cuda.synchronize()
    ref = oracle.gsd_verify_tree(wl.as_numpy_logits(inp["target"]), wl.as_numpy_logits(inp["draft"]), tok.cpu().numpy(),
                                 parent, wl.seeds_as_u64(inp["seeds"]), T=inp["T"])
    amb = ambiguous(ref)
    assert amb.sum() <= 1
    ok = ~amb
    assert (acc.cpu().numpy()[ok] == ref["accept_len"][ok]).all()
    assert (out.cpu().numpy()[ok] == ref["tokens"][ok]).all()
    assert (path.cpu().numpy()[ok] == ref["path"][ok]).all()


def test_gsd_and_ersd_acceptance_on_the_same_rows(ersd):
    """Section 3 on synthetic Zipf rows at vocabulary size: GSD accepts the first drafted token with
    probability 1 - D_TV, ERSD's match rate lies between D_HM and that (Lemma 3.1); summed over
    the rows of config 3's sigma = 1 point both counts fall within 4.5 sigma of those sums."""
    import math
    w = wl.scaled(wl.CONFIGS["c3"], B=64)
    inp = wl.make_inputs(w, call=1, sigma=1.0, T=1.0, device="cuda")
    tgt, drf, seeds = inp["target"], inp["draft"], inp["seeds"]
    res = ersd.verify(tgt, drf, seeds, 1.0)
    tok = draft_tokens(ersd, drf, seeds + 12345, 1.0)[..., 0].contiguous()     # drafted with races of their own
    out = torch.empty(w.B, w.k + 1, dtype=torch.int32, device="cuda")
    acc = torch.empty(w.B, dtype=torch.int32, device="cuda")
    ersd.ersd_gsd_verify(tgt, drf, tok, seeds, 1.0, out, acc)
    torch.cuda.synchronize()
    p = torch.softmax(tgt[:, 0].double(), -1)
    q = torch.softmax(drf[:, 0].double(), -1)
    a_gsd = (1.0 - 0.5 * (p - q).abs().sum(-1)).cpu().numpy()
    d_hm = (p * q / (p + q)).sum(-1).cpu().numpy()
    got_g = int((acc >= 1).sum().item())
    got_e = int((res["accept_len"] >= 1).sum().item())
    sd = math.sqrt((a_gsd * (1 - a_gsd)).sum())
    assert abs(got_g - a_gsd.sum()) < 4.5 * sd, (got_g, a_gsd.sum())
    assert d_hm.sum() - 4.5 * sd <= got_e <= a_gsd.sum() + 4.5 * sd, (got_e, d_hm.sum(), a_gsd.sum())


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [1, 7, 8, 9, 1023, 2049, 4099, 40001])
def test_sequence_gsd_rows_of_any_length(ersd, V, dtype):
    """Slices of less than one group, ragged ends, rows on every 16-byte offset, NaN and infinite logits."""
    w = wl.Workload("gsdlen", B=9, k=3, V=V, dtype=dtype, sigma=0.7, T=0.8, config_id=51)
    inp = wl.make_inputs(w)
    tok = draft_tokens(ersd, inp["draft"].cuda(), inp["seeds"].cuda(), inp["T"])[..., 0].contiguous()
    if V > 8:
        inp["target"][0, :, 1::3] = float("nan")
        inp["draft"][1, :, 2::3] = float("nan")
        inp["target"][2, :, V // 2:] = float("-inf")
        inp["draft"][3, :, : V // 2] = float("-inf")
        inp["target"][4, 1] = float("-inf")                     # a law without support
    out = torch.full((w.B, w.k + 1), -9, dtype=torch.int32, device="cuda")
    acc = torch.full((w.B,), -9, dtype=torch.int32, device="cuda")
    ersd.ersd_gsd_verify(inp["target"].cuda(), inp["draft"].cuda(), tok, inp["seeds"].cuda(), inp["T"], out, acc)
    torch.cuda.synchronize()
    ref = oracle.gsd_verify(wl.as_numpy_logits(inp["target"]), wl.as_numpy_logits(inp["draft"]), tok.cpu().numpy(),
                            wl.seeds_as_u64(inp["seeds"]), T=inp["T"])
    ok = ~ambiguous(ref)
    assert ok.sum() >= w.B - 1
    assert (acc.cpu().numpy()[ok] == ref["accept_len"][ok]).all()
    assert (out.cpu().numpy()[ok] == ref["tokens"][ok]).all()


@pytest.mark.parametrize("off", [-2e-6, 2e-6])
def test_ratio_tests_too_close_for_single_precision(ersd, off):
    """Ratios 2e-6 away from their uniform number, far inside what single-precision sums can tell
    (about 1e-5) and far outside what double precision cannot: every test takes the exact path."""
    B, V = 64, 5000
    g = torch.Generator().manual_seed(8)
    drf = torch.randn(B, 1, V, generator=g, dtype=torch.float64)
    x = torch.randint(0, V, (B, 1), generator=g)
    seeds = wl.make_seeds(21, 0, B)
    tok = x.to(torch.int32)
    tgt = torch.randn(B, 2, V, generator=g).float()
    first = oracle.gsd_verify(tgt.numpy(), drf.float().numpy(), tok.numpy(), wl.seeds_as_u64(seeds), T=1.0)
    drf = drf.float()
    d = drf[:, 0].double()
    q = torch.softmax(d, -1).gather(1, x)[:, 0]
    r = torch.from_numpy(first["unif"][:, 0]) * (1.0 + off)     # wanted ratio: the target law lifts or lowers token x alone
    z = d.gather(1, x)[:, 0] + torch.log(r * (1 - q) / (1 - r * q))
    t0 = d.clone()
    t0.scatter_(1, x, z.unsqueeze(1))
    tgt[:, 0] = t0.float()
    out = torch.empty(B, 2, dtype=torch.int32, device="cuda")
    acc = torch.empty(B, dtype=torch.int32, device="cuda")
    ersd.ersd_gsd_verify(tgt.cuda(), drf.cuda(), tok.cuda(), seeds.cuda(), 1.0, out, acc)
    torch.cuda.synchronize()
    ref = oracle.gsd_verify(tgt.numpy(), drf.numpy(), tok.numpy(), wl.seeds_as_u64(seeds), T=1.0)
    close = np.abs(ref["ratio"][:, 0] / ref["unif"][:, 0] - 1.0)
    assert close.max() < 6e-6 and not ambiguous(ref).any()      # (float32 logits: the ratio is off by their rounding)
    assert (acc.cpu().numpy() == ref["accept_len"]).all() and (out.cpu().numpy() == ref["tokens"]).all()


def test_final_races_too_close_for_single_precision(ersd):
    """Two tokens whose arrival times differ by 2e-5 relative: outside the near-tie window, inside the
    intervals of the single-precision race."""
    B, V = 64, 9000
    g = torch.Generator().manual_seed(9)
    tgt = torch.full((B, 1, V), float("-inf"))
    a, b = torch.randint(0, 4000, (B,), generator=g), torch.randint(4000, V, (B,), generator=g)
    n = torch.arange(B)
    tgt[n, 0, a] = 0.0
    tgt[n, 0, b] = 0.0
    seeds = wl.make_seeds(22, 0, B)
    none = np.zeros((B, 0), np.int32)
    ref = oracle.gsd_verify(tgt.numpy(), np.zeros((B, 0, V), np.float32), none, wl.seeds_as_u64(seeds), T=1.0)
    t, win = ref["last_times"], torch.from_numpy(ref["tokens"][:, 0].astype(np.int64))
    other = torch.where(win == a, b, a)
    tgt[n, 0, other] = torch.from_numpy(np.log(t[:, 1] / t[:, 0]) - 2e-5).float()    # the later one draws level
    ref = oracle.gsd_verify(tgt.numpy(), np.zeros((B, 0, V), np.float32), none, wl.seeds_as_u64(seeds), T=1.0)
    gap = ref["last_times"][:, 1] / ref["last_times"][:, 0] - 1.0
    ok = gap > 1e-5
    assert gap.max() < 4e-5 and ok.sum() > B // 2
    out = torch.empty(B, 1, dtype=torch.int32, device="cuda")
    acc = torch.empty(B, dtype=torch.int32, device="cuda")
    ersd.ersd_gsd_verify(tgt.cuda(), None, None, seeds.cuda(), 1.0, out, acc)
    torch.cuda.synchronize()
    assert (acc == 0).all() and (out.cpu().numpy()[ok] == ref["tokens"][ok]).all()


def test_long_drafts_that_end_in_exact_races(ersd):
    """More output columns than a warp has lanes, races decided by single and by double precision in
    neighbouring sequences: the last block of every sequence writes all its columns and leaves all of
    its scratch zeroed."""
    B, k, V = 48, 40, 600
    w = wl.Workload("gsdlong", B=B, k=k, V=V, dtype="f32", sigma=0.0, T=1.0, config_id=52)
    inp = wl.make_inputs(w)
    tok = draft_tokens(ersd, inp["draft"].cuda(), inp["seeds"].cuda(), inp["T"])[..., 0].contiguous()
    for b in range(0, B, 2):                                    # a law without support ends every other sequence
        inp["target"][b, (7 * b) % (k + 1)] = float("-inf")
    ref = oracle.gsd_verify(wl.as_numpy_logits(inp["target"]), wl.as_numpy_logits(inp["draft"]), tok.cpu().numpy(),
                            wl.seeds_as_u64(inp["seeds"]), T=inp["T"])
    ok = ~ambiguous(ref)
    assert ok.sum() >= B - 1 and (ref["accept_len"] == k).sum() >= B // 4
    tgt, drf, seeds = inp["target"].cuda(), inp["draft"].cuda(), inp["seeds"].cuda()
    ws = torch.empty(ersd.ersd_workspace_bytes(B, k + 1), dtype=torch.uint8, device="cuda")
    ersd.ersd_workspace_init(ws)
    for rep in range(5):
        out = torch.full((B, k + 1), -9, dtype=torch.int32, device="cuda")
        acc = torch.full((B,), -9, dtype=torch.int32, device="cuda")
        ersd.ersd_gsd_verify(tgt, drf, tok, seeds, inp["T"], out, acc, ersd.make_opts(workspace=ws))
        torch.cuda.synchronize()
        assert (ws == 0).all(), rep
        assert (acc.cpu().numpy()[ok] == ref["accept_len"][ok]).all()
        assert (out.cpu().numpy()[ok] == ref["tokens"][ok]).all()


@pytest.mark.parametrize("T", [1.0, 0.25])
def test_tokens_whose_probability_is_nothing_in_double_precision(ersd, T):
    """Given tokens with log2 probabilities from -8 down past the end of double precision's range (2^-1075)
    and at -inf, under either law, in every combination: ratios of 0, of infinity, 0/0 and ordinary ones.
    (Between -1080 and -1020, where a probability loses its digits, two exponentials may differ.)"""
    grid = [float("-inf"), -3000, -1200, -1160, -1140, -1100, -1010, -950, -905, -895, -500, -60, -8]
    B, V = len(grid) ** 2, 500
    g = torch.Generator().manual_seed(10)
    drf = torch.randn(B, 1, V, generator=g)
    tgt = torch.randn(B, 2, V, generator=g)
    x = torch.randint(0, V, (B,), generator=g)
    n = torch.arange(B)
    for rows, which in ((tgt, n // len(grid)), (drf, n % len(grid))):
        rest = rows[:, 0].double() / T
        rest[n, x] = float("-inf")
        lp = torch.tensor(grid, dtype=torch.float64)[which] * np.log(2.0)
        rows[n, 0, x] = ((torch.logsumexp(rest, -1) + lp) * T).float()
    tok = x.view(B, 1).to(torch.int32)
    seeds = wl.make_seeds(23, 0, B)
    out = torch.full((B, 2), -9, dtype=torch.int32, device="cuda")
    acc = torch.full((B,), -9, dtype=torch.int32, device="cuda")
    ersd.ersd_gsd_verify(tgt.cuda(), drf.cuda(), tok.cuda(), seeds.cuda(), T, out, acc)
    torch.cuda.synchronize()
    ref = oracle.gsd_verify(tgt.numpy(), drf.numpy(), tok.numpy(), wl.seeds_as_u64(seeds), T=T)
    ok = ~ambiguous(ref)
    assert ok.sum() >= B - 1 and len(grid) < ref["accept_len"].sum() < B - len(grid)
    assert (acc.cpu().numpy()[ok] == ref["accept_len"][ok]).all()
    assert (out.cpu().numpy()[ok] == ref["tokens"][ok]).all()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [7, 40001, 128256])
def test_rows_that_are_no_law(ersd, V, dtype):
    """A logit of +inf (the drafted token's or another one's), or none above -inf, in the target row, the
    draft row or the last row: nothing is accepted there and nothing emitted; and the masked token of an
    ordinary row."""
    B, k = 12, 3
    w = wl.Workload("gsdlaw", B=B, k=k, V=V, dtype=dtype, sigma=0.3, T=0.9, config_id=53)
    inp = wl.make_inputs(w)
    tgt, drf, inf = inp["target"], inp["draft"], float("inf")
    tok = draft_tokens(ersd, drf.cuda(), inp["seeds"].cuda(), inp["T"])[..., 0].contiguous()
    x = tok.cpu().long()
    tgt[0, 0, x[0, 0]] = inf
    tgt[1, 1, V // 2] = inf
    drf[2, 0, x[2, 0]] = inf
    drf[3, 2, V - 1] = inf
    tgt[4, k, 0] = inf
    tgt[5, k] = -inf
    tgt[6, 0] = -inf
    drf[7, 0] = -inf
    tgt[8, 0, x[8, 0]] = -inf
    drf[9, 0, x[9, 0]] = -inf
    tgt[10, 0, :] = float("nan")
    tgt[11, 0, 1:] = -inf
    out = torch.full((B, k + 1), -9, dtype=torch.int32, device="cuda")
    acc = torch.full((B,), -9, dtype=torch.int32, device="cuda")
    for rep in range(2):
        ersd.ersd_gsd_verify(tgt.cuda(), drf.cuda(), tok, inp["seeds"].cuda(), inp["T"], out, acc)
    torch.cuda.synchronize()
    ref = oracle.gsd_verify(wl.as_numpy_logits(tgt), wl.as_numpy_logits(drf), tok.cpu().numpy(),
                            wl.seeds_as_u64(inp["seeds"]), T=inp["T"])
    ok = ~ambiguous(ref)
    assert ok.sum() >= B - 1
    assert (acc.cpu().numpy()[ok] == ref["accept_len"][ok]).all()
    assert (out.cpu().numpy()[ok] == ref["tokens"][ok]).all()


def test_masked_and_infinite_logits_take_no_second_reading(ersd):
    """A drafted token that the target's mask rules out, and a row with a logit of +inf, are decided by the
    sums that every call takes.  (Read again in double precision by one block such a call took 153 and 530 us,
    an ordinary one 14: a factor of three leaves room for a disturbed clock.)"""
    w = wl.scaled(wl.CONFIGS["c5"], B=1)
    inp = wl.make_inputs(w, device="cuda")
    tgt, drf, seeds = inp["target"], inp["draft"], inp["seeds"]
    tok = draft_tokens(ersd, drf, seeds, 1.0)[..., 0].contiguous()
    masked, infinite = tgt.clone(), tgt.clone()
    masked[0, 0, tok[0, 0].item()] = float("-inf")
    infinite[0, 0, 5] = float("inf")
    out = torch.empty(1, w.k + 1, dtype=torch.int32, device="cuda")
    acc = torch.empty(1, dtype=torch.int32, device="cuda")

    def us(t):
        best = float("inf")
        for rep in range(12):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for q in range(20):
                ersd.ersd_gsd_verify(t, drf, tok, seeds, 1.0, out, acc)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1) * 50.0)
        return best

    plain = us(tgt)
    assert us(masked) < 3.0 * plain and us(infinite) < 3.0 * plain


@pytest.mark.parametrize("T", [0.05, 0.2])
@pytest.mark.parametrize("V", [3001, 40000])
def test_tokens_drafted_at_another_temperature(ersd, V, T):
    """Given tokens that the laws at a low temperature would hardly draw: rejected, and then the residual
    hangs on the last digits of one token's two probabilities, so the last race is run in double precision.
    A difference of less than 1e-9 of them is left out: both are known to a few 2^-53, so its own error passes
    1e-6, a tenth of the window inside which two arrivals may come either way."""
    B, k = 64, 2
    w = wl.Workload("gsdcold", B=B, k=k, V=V, dtype="bf16", sigma=0.3, T=T, config_id=54)
    inp = wl.make_inputs(w)
    tok = draft_tokens(ersd, inp["draft"].cuda(), inp["seeds"].cuda(), 1.0)[..., 0].contiguous()
    out = torch.full((B, k + 1), -9, dtype=torch.int32, device="cuda")
    acc = torch.full((B,), -9, dtype=torch.int32, device="cuda")
    ersd.ersd_gsd_verify(inp["target"].cuda(), inp["draft"].cuda(), tok, inp["seeds"].cuda(), T, out, acc)
    torch.cuda.synchronize()
    ref = oracle.gsd_verify(wl.as_numpy_logits(inp["target"]), wl.as_numpy_logits(inp["draft"]), tok.cpu().numpy(),
                            wl.seeds_as_u64(inp["seeds"]), T=T)
    n, L = np.arange(B), np.minimum(ref["accept_len"], k - 1)
    p = torch.softmax(inp["target"][n, L].double() / T, -1)
    q = torch.softmax(inp["draft"][n, L].double() / T, -1)
    either = torch.maximum(p, q)
    close = ((either > 1e-3) & ((p - q).abs() < 1e-9 * either)).any(-1).numpy()
    ok = ~ambiguous(ref) & ~close
    assert ok.sum() >= B // 2 and (ref["accept_len"] == 0).sum() >= B // 4
    assert (acc.cpu().numpy()[ok] == ref["accept_len"][ok]).all()
    assert (out.cpu().numpy()[ok] == ref["tokens"][ok]).all()


@pytest.mark.parametrize("k,V", [(31, 900), (32, 1025), (127, 1025), (128, 3000), (200, 1000), (255, 40), (60, 40000)])
def test_long_drafts_of_short_rows(ersd, k, V):
    """Rows of one slice and of several, more rows than a block's warps or lanes take at a time, runs of
    accepted tokens that end in the middle of 32, at their end and at the last row."""
    B = 6
    w = wl.Workload("gsdrun", B=B, k=k, V=V, dtype="f32", sigma=0.02, T=1.0, config_id=55)
    inp = wl.make_inputs(w)
    tok = draft_tokens(ersd, inp["draft"].cuda(), inp["seeds"].cuda(), inp["T"])[..., 0].contiguous()
    inp["draft"][0] = inp["target"][0, :k]                      # (all accepted)
    inp["target"][1, 31 % k] = float("-inf")
    inp["target"][2, min(32, k - 1)] = float("-inf")
    out = torch.full((B, k + 1), -9, dtype=torch.int32, device="cuda")
    acc = torch.full((B,), -9, dtype=torch.int32, device="cuda")
    ersd.ersd_gsd_verify(inp["target"].cuda(), inp["draft"].cuda(), tok, inp["seeds"].cuda(), inp["T"], out, acc)
    torch.cuda.synchronize()
    ref = oracle.gsd_verify(wl.as_numpy_logits(inp["target"]), wl.as_numpy_logits(inp["draft"]), tok.cpu().numpy(),
                            wl.seeds_as_u64(inp["seeds"]), T=inp["T"])
    ok = ~ambiguous(ref)
    assert ok.sum() >= B - 1 and ref["accept_len"][0] == k
    assert (acc.cpu().numpy()[ok] == ref["accept_len"][ok]).all()
    assert (out.cpu().numpy()[ok] == ref["tokens"][ok]).all()
