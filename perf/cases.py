"""What this library is timed on: the calls that a decoding loop makes, from one drafted token to a
serving-size verification.

A case names the entry point (``call``), the sizes, the storage type of the logits and the options.
Inputs follow the recipe of ``workloads.py`` (Zipf-shaped rows, draft rows = target rows + noise);
buffers for the results and the options structure are made once, as a decoding loop keeps them.
"""
from __future__ import annotations

import math

import torch

from paper_2504_15475_b200 import binding, workloads as wl

# draft trees by name: the two of workloads.py, and batch drafting (k alternatives for one position)
TREES = {"4x4": list(wl.TREE_4x4), "specinfer": list(wl.TREE_SPECINFER), "star4": wl.star_parent(4),
         "star8": wl.star_parent(8)}
TEMPS = (0.6, 0.8, 1.0)  # temps="mixed": one temperature per sequence out of these


def _case(name, call, B, V, k=0, **more):
    c = dict(name=name, call=call, B=B, k=k, V=V, dtype="bf16", top_c=1, tree="", T=1.0, temps="one",
             zipf=1.1, sigma=1.0, rows=False)
    c.update(more)
    return c


def listed():
    return [
        # drafting: the next token of one sequence, as the draft model's loop asks for it k times per round
        _case("draft_1", "sample", B=1, V=128256),
        # batch drafting: eight alternatives for each of four sequences, with their race keys
        _case("draft_top8_4", "sample", B=4, V=128256, top_c=8, rows=True),
        # one sequence decoded at a time (how the paper's experiments run), five drafted tokens
        _case("verify_1", "verify", B=1, V=128256, k=5),
        # the same with a draft tree of four candidates extended to depth four
        _case("tree_1", "tree", B=1, V=128256, tree="4x4", rows=True),
        # a few sequences over a vocabulary of 32000
        _case("verify_8_v32000", "verify", B=8, V=32000, k=4, sigma=0.5, rows=True),
        # the same vocabulary with one token added: no row but the first starts on a 16-byte boundary
        _case("verify_16_v32001", "verify", B=16, V=32001, k=4, rows=True),
        # an ordinary serving batch
        _case("verify_24", "verify", B=24, V=128256, k=5, temps="mixed"),
        # single-precision logits, tokens drafted earlier by the draft model's own loop
        _case("tokens_48_f32", "tokens", B=48, V=128256, k=4, dtype="f32", temps="mixed", rows=True),
        # a larger batch with long drafts, every row's winner and key wanted (acceptance statistics)
        _case("verify_64", "verify", B=64, V=128256, k=8, rows=True),
        # tree drafting in a serving batch
        _case("tree_32", "tree", B=32, V=151936, tree="4x4", rows=True),
        # the paper's comparison verifier on an ordinary batch
        _case("gsd_64", "gsd", B=64, V=128256, k=5),
        # serving scale: 256 sequences with temperatures of their own
        _case("verify_256", "verify", B=256, V=128256, k=5, temps="mixed", rows=True),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rows_read(c):
    """Logit rows of one sequence that the call reads."""
    if c["call"] == "sample":
        return 1
    if c["call"] == "tokens":
        return c["k"] + 1
    if c["call"] == "tree":
        parent = TREES[c["tree"]]
        return len(parent) + len({p for p in parent if p >= 0})
    return 2 * c["k"] + 1


def _logit_bytes(c):
    return c["B"] * _rows_read(c) * c["V"] * (2 if c["dtype"] == "bf16" else 4)


def draw(rng):
    call = rng.choice(("sample", "sample", "verify", "verify", "verify", "tokens", "tree", "gsd"))
    c = _case("", call, B=1, V=1)
    del c["name"]
    # half of the vocabularies are the sizes of the configurations, half any size (mostly not a multiple of eight)
    c["V"] = rng.choice((32000, 128256, 151936)) if rng.random() < 0.5 else _log_uniform(rng, 1000, 152000)
    c["dtype"] = rng.choice(("bf16", "bf16", "bf16", "f32"))
    c["sigma"] = rng.choice((0.25, 0.5, 1.0, 2.0))
    c["zipf"] = round(rng.uniform(0.9, 1.3), 3)
    c["rows"] = rng.random() < 0.5
    if rng.random() < 0.3:
        c["temps"] = "mixed"
    else:
        c["T"] = rng.choice((0.6, 0.7, 0.8, 1.0, 1.0)) if call == "gsd" else rng.choice((0.0, 0.6, 0.7, 1.0, 1.0))
    if call == "sample":
        c["top_c"] = rng.choice((1, 1, 2, 4, 8))
        most = 256
    elif call == "tree":
        c["tree"] = rng.choice(sorted(TREES))
        most = 64
    else:
        c["k"] = rng.randint(1, 8)
        most = 64 if call == "gsd" else 256
    c["B"] = _log_uniform(rng, 1, most)
    # no call larger than the largest listed one of its kind
    limit = {"gsd": 64 * 11 * 128256 * 2, "tree": 32 * 30 * 151936 * 2}.get(call, 256 * 11 * 128256 * 2)
    while c["B"] > 1 and _logit_bytes(c) > limit:
        c["B"] -= 1
    return c


def prepare(case, seed):
    c = case
    parent = TREES[c["tree"]] if c["call"] == "tree" else None
    if c["call"] == "sample":
        k = 0
    elif parent is not None:
        k = len(parent) - 1
    else:
        k = c["k"]
    w = wl.Workload("case", B=c["B"], k=k, V=c["V"], dtype=c["dtype"], sigma=c["sigma"], T=c["T"], zipf=c["zipf"],
                    temps_choices=TEMPS if c["temps"] == "mixed" else None,
                    parent=None if parent is None else tuple(parent))
    s = dict(wl.make_inputs(w, call=seed, device="cuda"), call=c["call"])
    B, rows = c["B"], k + 1

    def new(*shape, dtype=torch.int32):
        return torch.zeros(*shape, dtype=dtype, device="cuda")

    opts = {}
    if s["temps"] is not None:
        opts.update(temps=s["temps"], temp_strides=(s["temps"].stride(0), s["temps"].stride(1)))
    # where each sequence's text stands: the races of a decoding loop are keyed by it
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s["positions"] = torch.randint(0, 4096, (B,), generator=gen, device="cuda", dtype=torch.int32)
    opts.update(pos_offsets=s["positions"])

    if c["call"] in ("tokens", "gsd"):
        # the tokens that the draft model's loop drafted, one position at a time
        drafted = new(B, k, 1)
        temps = {}
        if s["temps"] is not None:
            s["draft_temps"] = s["temps"][:, :k].contiguous()
            temps = dict(temps=s["draft_temps"], temp_strides=(s["draft_temps"].stride(0), s["draft_temps"].stride(1)))
        binding.ersd_race_sample(s["draft"], s["seeds"], s["T"], drafted,
                                 binding.make_opts(pos_offsets=s["positions"], **temps))
        s["drafted"] = drafted.view(B, k)
        if c["call"] == "tokens":
            del s["draft"]

    if c["call"] == "sample":
        out = {"tok": new(B, 1, c["top_c"])}
        if c["rows"]:
            out["key"] = new(B, 1, c["top_c"], dtype=torch.float32)
            opts.update(out_key=out["key"])
        opts.update(top_c=c["top_c"])
    else:
        depth = k if parent is None else binding.ersd_tree_depth(parent)
        out = {"tokens": new(B, depth + 1), "accept": new(B)}
        if parent is not None:
            out["path"] = new(B, depth + 1)
            opts.update(out_path=out["path"])
        if c["rows"] and c["call"] != "gsd":
            out["target_tok"], out["target_key"] = new(B, rows), new(B, rows, dtype=torch.float32)
            opts.update(out_target_tok=out["target_tok"], out_target_key=out["target_key"])
            if c["call"] != "tokens":
                drafts = rows if parent is not None else k
                out["draft_tok"], out["draft_key"] = new(B, drafts), new(B, drafts, dtype=torch.float32)
                opts.update(out_draft_tok=out["draft_tok"], out_draft_key=out["draft_key"])
    s["out"] = out
    s["opts"] = binding.make_opts(**opts)
    return s


def run(state):
    s, out = state, state["out"]
    call = s["call"]
    if call == "sample":
        binding.ersd_race_sample(s["target"], s["seeds"], s["T"], out["tok"], s["opts"])
    elif call == "verify":
        binding.ersd_verify(s["target"], s["draft"], s["seeds"], s["T"], out["tokens"], out["accept"], s["opts"])
    elif call == "tokens":
        binding.ersd_verify_tokens(s["target"], s["drafted"], s["seeds"], s["T"], out["tokens"], out["accept"],
                                   s["opts"])
    elif call == "tree":
        binding.ersd_verify_tree(s["target"], s["draft"], s["parent"], s["seeds"], s["T"], out["tokens"],
                                 out["accept"], s["opts"])
    else:
        binding.ersd_gsd_verify(s["target"], s["draft"], s["drafted"], s["seeds"], s["T"], out["tokens"],
                                out["accept"], s["opts"])
    return out


def work(case):
    """Every logit row read once; per vocabulary index of a race a quarter of a Philox4x32-10 call (9.25
    integer operations) and a multiply-add per logit."""
    c = case
    races = {"sample": 1, "tree": len(TREES.get(c["tree"], ()))}.get(c["call"], c["k"] + 1)
    if c["call"] == "gsd":
        races = 1  # the race that draws the last token; the ratio tests draw one number each
    per_logit = 4 if c["call"] == "gsd" else 2  # (the softmax's exponential and sum)
    out = 8 * c["B"] * (_rows_read(c) + c["top_c"])
    return {"bytes": _logit_bytes(c) + out,
            "flops": c["B"] * c["V"] * (races * 9.25 + _rows_read(c) * per_logit)}


def tolerance(case):
    # Tokens, lengths and paths are whole numbers and the same for every correct implementation (decisions are
    # taken in double precision).  Race keys are double-precision values rounded to single precision: at most one
    # rounding apart (6e-8 of the value, two of them 1.2e-7).
    return {"rel": 2e-7, "max": 4e-7, "differ": 0.0}
