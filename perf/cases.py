"""Workloads for measuring the framework through its public entry points.

Every case is a call (or a short run of calls) that a program using the
framework makes: whole joins, the graph-captured batch of joins, EmbedJoin+,
search against a resident index, and the per-stage calls. Inputs have the
shapes of ``paper_1702_00093_gb300.synth`` (clustered DNA, protein-like and
text-like sets, a serving index with queries), drawn on the GPU so that large
sets are made quickly. Outputs are sorted pair lists and signature keys, all
whole numbers.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1702_00093_gb300 import embedjoin as ej
from paper_1702_00093_gb300 import synth

DEVICE = "cuda:0"
SEED = 1   # of the method's random strings and positions


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
# Fields: do = the call; shape = dna | protein | text; n = strings; len =
# typical string length; K = threshold; r, m, z, L = method parameters (L = 0:
# the library's own sampling range); host = strings and result in host memory.

def listed() -> list:
    return [
        # an interactive join of a thousand short reads: launches and host
        # round trips are all of it
        dict(name="join_dna_small", do="join", shape="dna", n=1000, len=100, K=6, r=3, m=10, z=12, L=0, host=False),
        # the headline shape: long reads at 3% distance, few candidates
        dict(name="join_dna_long", do="join", shape="dna", n=20000, len=5000, K=150, r=7, m=20, z=14, L=5000,
             host=False),
        # long reads with few samples per function: high recall, millions of
        # candidates, the verifier's throughput
        dict(name="join_dna_recall", do="join", shape="dna", n=20000, len=5000, K=250, r=7, m=20, z=7, L=5000,
             host=False),
        # several thresholds over one set, replayed as one CUDA graph
        dict(name="batch_dna_long", do="batch", shape="dna", n=20000, len=5000, K=250, r=7, m=20, z=13, L=5000,
             host=False),
        # a protein collection at full size: a 25-letter alphabet, short strings
        # of very different lengths, hundreds of millions of candidates
        dict(name="join_protein", do="join", shape="protein", n=200000, len=400, K=40, r=7, m=7, z=8, L=890,
             host=False),
        # abstracts: 37 symbols, up to 3000 characters, clusters of near-duplicates
        dict(name="join_text", do="join", shape="text", n=120000, len=1900, K=200, r=7, m=7, z=9, L=3800, host=False),
        # a small odd-sized set whose strings and result live in host memory
        dict(name="join_protein_host", do="join", shape="protein", n=5003, len=400, K=60, r=7, m=7, z=8, L=890,
             host=True),
        # EmbedJoin+ on long reads (shifted alignments)
        dict(name="join_plus_dna", do="plus", shape="dna", n=20000, len=5000, K=150, r=7, m=16, z=14, L=5000,
             host=False),
        # one query against a resident index: the latency a service pays
        dict(name="search_one", do="search", shape="dna", n=300000, len=1000, queries=1, r=7, m=7, z=8, L=1000,
             host=True),
        # a bulk search of many queries of mixed lengths and thresholds
        dict(name="search_many", do="search", shape="dna", n=300000, len=1000, queries=2000, r=7, m=7, z=8, L=1000,
             host=True),
        # the stages one by one (keys, candidates, verification), as a program
        # that keeps or filters the intermediate results calls them
        dict(name="stages_dna", do="stages", shape="dna", n=20000, len=5000, K=150, r=7, m=20, z=14, L=5000,
             host=False),
        dict(name="stages_text", do="stages", shape="text", n=30011, len=1900, K=100, r=7, m=7, z=10, L=3800,
             host=False),
    ]


def _log_int(rng: random.Random, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random) -> dict:
    do = rng.choice(["join", "join", "join", "batch", "plus", "search", "stages"])
    shape = rng.choice(["dna", "protein", "text"]) if do in ("join", "stages") else "dna"
    host = do == "join" and rng.random() < 0.3
    if do == "search":
        return dict(do=do, shape=shape, n=_log_int(rng, 5000, 300000), len=1000, queries=_log_int(rng, 1, 2000), r=7,
                    m=7, z=8, L=1000, host=True)
    if shape == "protein":
        K = rng.randint(20, 60)
        return dict(do=do, shape=shape, n=_log_int(rng, 1000, 100000 if do == "join" else 20000), len=400, K=K, r=7,
                    m=7, z=8, L=890, host=host)
    if shape == "text":
        K = rng.randint(50, 300)
        return dict(do=do, shape=shape, n=_log_int(rng, 1000, 60000 if do == "join" else 20000), len=1900, K=K, r=7,
                    m=7, z=10 if K <= 100 else 9, L=3800, host=host)
    length = _log_int(rng, 100, 5000)
    K = max(1, int(round(rng.uniform(0.01, 0.05) * length)))
    x = 100.0 * K / length
    z = max(9, int(round(math.log2(length))) + 3 - int(math.floor(math.log2(x))))
    if do == "join" and length >= 2000 and rng.random() < 0.3:
        z = rng.randint(8, 10)   # high recall
    return dict(do=do, shape=shape, n=_log_int(rng, 500, 20000), len=length, K=K, r=rng.choice([3, 5, 7]),
                m=rng.randint(8, 20), z=z, L=length, host=host)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

_ALPHABET = {"dna": synth.DNA, "protein": synth.PROTEIN, "text": synth.TEXT}


def _frequencies(shape: str) -> np.ndarray:
    if shape == "protein":
        return synth.zipf_freqs(25, 1.0)
    if shape == "text":
        return synth.text_freqs()
    return np.full(4, 0.25)


def _symbols(count: int, shape: str, g: torch.Generator) -> torch.Tensor:
    """Symbol codes drawn independently with the shape's frequencies."""
    if shape == "dna":
        return torch.randint(0, 4, (count,), generator=g, device=DEVICE, dtype=torch.uint8)
    edges = torch.from_numpy(np.cumsum(_frequencies(shape))[:-1].astype(np.float32)).to(DEVICE)
    u = torch.rand(count, generator=g, device=DEVICE)
    return torch.bucketize(u, edges, out_int32=True, right=True).to(torch.uint8)


def _offsets(lens: torch.Tensor) -> torch.Tensor:
    o = torch.zeros(lens.numel() + 1, dtype=torch.int64, device=DEVICE)
    torch.cumsum(lens, 0, out=o[1:])
    return o


def _mutated(src: torch.Tensor, rate: torch.Tensor, base: torch.Tensor, boff: torch.Tensor, shape: str,
             g: torch.Generator):
    """Codes and offsets of copies of the base strings src[i], every position of
    copy i edited with probability rate[i] (substitution, deletion or insertion,
    equally likely)."""
    sigma = len(_ALPHABET[shape])
    lens = (boff[1:] - boff[:-1])[src]
    soff = _offsets(lens)
    total = int(soff[-1])
    owner = torch.repeat_interleave(torch.arange(src.numel(), device=DEVICE, dtype=torch.int32), lens,
                                    output_size=total)
    at = torch.arange(total, device=DEVICE) + (boff[:-1][src] - soff[:-1])[owner]
    sym = base[at]
    del at
    u = torch.rand(total, generator=g, device=DEVICE) / rate.clamp_min(1e-9)[owner]   # < 1: an edit
    edit = torch.where(rate[owner] > 0, u, 2.0)
    del u, owner
    sub, dele, ins = edit < 1 / 3, (edit >= 1 / 3) & (edit < 2 / 3), (edit >= 2 / 3) & (edit < 1)
    del edit
    shift = torch.randint(1, sigma, (total,), generator=g, device=DEVICE, dtype=torch.uint8)
    sym = torch.where(sub, (sym + shift) % sigma, sym)
    del shift, sub
    count = torch.ones(total, dtype=torch.int8, device=DEVICE) + ins.to(torch.int8) - dele.to(torch.int8)
    end = torch.cumsum(count, 0, dtype=torch.int64)
    out = _symbols(int(end[-1]) if total else 0, shape, g)   # the inserted symbols stay as drawn
    keep = ~dele
    out[end[keep] - 1] = sym[keep]
    off = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEVICE), end])[soff]
    return out, off


def _lengths(count: int, case: dict, g: torch.Generator) -> torch.Tensor:
    mean = float(case["len"])
    if case["shape"] == "protein":
        ln = torch.randn(count, generator=g, device=DEVICE) * 0.46 + math.log(mean)
        return ln.exp().round().clamp(mean / 4, mean * 5).to(torch.int64)
    lo, hi = (mean * 800 / 1900, mean * 3000 / 1900) if case["shape"] == "text" else (mean * 0.9, mean * 1.1)
    return torch.randint(int(lo), int(hi) + 1, (count,), generator=g, device=DEVICE)


def _set(case: dict, g: torch.Generator):
    """Codes and offsets of one string set with its shape's near-duplicates."""
    n, shape = case["n"], case["shape"]
    if shape == "protein" or case["do"] == "search":
        # mostly unrelated strings, some of them near-duplicates of others
        n_dup = n // 5 if shape == "protein" else n // 10
        base_n = n - n_dup
        src = torch.cat([torch.arange(base_n, device=DEVICE),
                         torch.randint(0, base_n, (n_dup,), generator=g, device=DEVICE)])
        rate = torch.zeros(n, device=DEVICE)
        rate[base_n:] = 0.05 if shape == "protein" else torch.rand(n_dup, generator=g, device=DEVICE) * 0.04 + 0.01
    else:
        # clusters: 10 reads, or 2 to 20 texts (11 on average), of one base each
        per = 10 if shape == "dna" else 11
        base_n = max(1, n // per)
        if shape == "dna":
            src = torch.arange(n, device=DEVICE) % base_n
        else:
            weight = torch.randint(2, 21, (base_n,), generator=g, device=DEVICE).to(torch.float32)
            src = torch.multinomial(weight, n, replacement=True, generator=g)
        lo, hi = (0.01, 0.08) if shape == "dna" else (0.02, 0.20)
        rate = torch.rand(n, generator=g, device=DEVICE) * (hi - lo) + lo
    mix = torch.randperm(n, generator=g, device=DEVICE)
    src, rate = src[mix], rate[mix]
    blen = _lengths(base_n, case, g)
    boff = _offsets(blen)
    base = _symbols(int(boff[-1]), shape, g)
    return _mutated(src, rate, base, boff, shape, g)


def _bytes(codes: torch.Tensor, shape: str) -> torch.Tensor:
    return torch.tensor(list(_ALPHABET[shape]), dtype=torch.uint8, device=DEVICE)[codes.to(torch.int32)]


def _params(case: dict, K: int | None = None, z: int | None = None) -> ej.Params:
    return ej.Params(K=case.get("K", 0) if K is None else K, r=case["r"], m=case["m"], z=case["z"] if z is None else z,
                     L=case["L"], seed=SEED, alphabet=_ALPHABET[case["shape"]])


def _queries(case: dict, codes: torch.Tensor, off: torch.Tensor, g: torch.Generator):
    """Half edited copies of index strings (rate 1% to 10%) whose threshold covers
    their edits, half fresh strings of a fifth to five times the index's length
    with K = 1% to 10% of it."""
    q = case["queries"]
    edited = (q + 1) // 2
    src = torch.randint(0, off.numel() - 1, (edited,), generator=g, device=DEVICE)
    rate = torch.rand(edited, generator=g, device=DEVICE) * 0.09 + 0.01
    qc, qo = _mutated(src, rate, codes, off, "dna", g)
    fresh = torch.randint(case["len"] // 5, case["len"] * 5 + 1, (q - edited,), generator=g, device=DEVICE)
    fc = _symbols(int(fresh.sum()) if q > edited else 0, "dna", g)
    lens = torch.cat([qo[1:] - qo[:-1], fresh])
    share = torch.rand(q, generator=g, device=DEVICE) * 0.09 + 0.01
    share[:edited] = rate + 0.02
    data = _bytes(torch.cat([qc, fc]), "dna").cpu().numpy()
    return ej.Strings(data, _offsets(lens).cpu().numpy()), (lens * share).round().to(torch.int32).cpu().numpy()


def _room(case: dict) -> int:
    """Entries of a result buffer: a few per string (a near-duplicate set has up
    to a cluster's size per string)."""
    return max(4096, 10 * case["n"])


def prepare(case: dict, seed: int) -> dict:
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed * 1000003 + 17)
    codes, off = _set(case, g)
    data = _bytes(codes, case["shape"])
    state = dict(do=case["do"], ctx=ej.Context(0), params=_params(case))
    if case["do"] == "search":
        strings = ej.Strings(data, off)
        state["index"] = ej.Index(state["ctx"], strings, state["params"])
        state["queries"], state["K"] = _queries(case, codes, off, g)
        state["found"] = np.zeros(max(64, 64 * case["queries"]), dtype=np.uint64)
        return state
    if case["host"]:
        state["strings"] = ej.Strings(data.cpu().numpy(), off.cpu().numpy())
        state["out"] = np.zeros(_room(case), dtype=np.uint64)
        return state
    state["strings"] = ej.Strings(data, off)
    room = _room(case)
    if case["do"] == "batch":
        # the set at a fifth, three fifths and all of K (long reads: 50 / 150 / 250)
        Ks = sorted({max(1, case["K"] // 5), max(1, case["K"] * 3 // 5), case["K"]})
        ps = [_params(case, K=k, z=case["z"] + len(Ks) - 1 - i) for i, k in enumerate(Ks)]
        state["outs"] = [torch.zeros(room, dtype=torch.int64, device=DEVICE) for _ in ps]
        state["stream"] = torch.cuda.Stream()
        state["stream"].wait_stream(torch.cuda.current_stream())
        state["batch"] = state["ctx"].batch(state["strings"], ps, stream=state["stream"])
        return state
    if case["do"] == "plus":
        state["delta"] = max(1, int(round(math.sqrt(case["len"]))))
    if case["do"] == "stages":
        # short and padded signatures collide often outside DNA: room by the square
        room = max(1 << 20, 40 * case["n"])
        if case["shape"] != "dna":
            room = max(room, case["n"] ** 2 // (16 if case["shape"] == "protein" else 64))
        state["keys"] = torch.zeros(case["r"] * case["m"] * case["n"], dtype=torch.int64, device=DEVICE)
        state["pairs"] = torch.zeros(room, dtype=torch.int64, device=DEVICE)
    state["out"] = torch.zeros(room, dtype=torch.int64, device=DEVICE)
    return state


# ---------------------------------------------------------------------------
# One pass: the call's counts, and its result buffers (zero beyond the counts)
# ---------------------------------------------------------------------------

def run(state: dict):
    do, ctx, p = state["do"], state["ctx"], state["params"]
    if do == "search":
        got = state["index"].search(state["queries"], state["K"])
        state["found"][:len(got)] = got
        return [len(got), state["found"]]
    if do == "batch":
        b, s = state["batch"], state["stream"]
        b.run(s)
        return [[b.result_into(i, out, stream=s)[0], out] for i, out in enumerate(state["outs"])]
    if do == "join":
        return [ctx.join_into(state["strings"], p, state["out"])[0], state["out"]]
    if do == "plus":
        T = 2 if p.K > state["delta"] else 1
        return [ctx.join_plus_into(state["strings"], p, state["delta"], T, state["out"])[0], state["out"]]
    s, keys, pairs = state["strings"], state["keys"], state["pairs"]
    ctx.embed_sign(s, p, keys)
    n, _ = ctx.lsh_candidates(s, p, keys, pairs)
    kept = ctx.verify(s, p, pairs[:n], state["out"])
    return [n, kept, keys, pairs, state["out"]]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def work(case: dict) -> dict:
    """Bytes: the strings and offsets read once, the result written once. Integer
    operations: one step of every walk per character (4 operations), and the
    band of every planted near-duplicate pair in 64-bit words (26 operations per
    word and column)."""
    n, length, shape = case["n"], case["len"], case["shape"]
    if case["do"] == "search":
        q = case["queries"]
        qlen = length * (0.5 * 1.0 + 0.5 * 2.6)
        hits = q * 0.3
        return dict(bytes=q * (qlen + 12) + hits * (length / 4 + 8),
                    flops=q * qlen * case["r"] * 4.0 + hits * length * math.ceil((0.055 * length + 1) / 64) * 26.0)
    mean = length * {"dna": 1.0, "protein": 1.11, "text": 1.0}[shape]
    pairs = n * {"dna": 4.5 * 0.2, "protein": 0.2, "text": 6.0 * 0.1}[shape]
    joins = 3 if case["do"] == "batch" else 1
    read = n * mean + 8.0 * (n + 1)
    out = 8.0 * pairs * joins
    if case["do"] == "stages":
        out += 8.0 * case["r"] * case["m"] * n + 16.0 * pairs
    suffixes = max(1, math.ceil(case["K"] / round(math.sqrt(length)))) if case["do"] == "plus" else 1
    walks = suffixes * n * case["r"] * min(mean, case["L"] / 1.5 if case["L"] else mean)
    return dict(bytes=read + out, flops=walks * 4.0 + pairs * mean * math.ceil((case["K"] + 1) / 64) * 26.0)


def exact(case: dict, seed: int):
    """Outputs are whole numbers (pair lists and keys), the same on every run."""
    return None
