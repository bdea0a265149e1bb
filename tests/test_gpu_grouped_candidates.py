"""Candidates grouped for the shared-string verifier against the hashed and sorted
paths with a pair-set deduplication: the same raw pairs, candidates, largest bucket
and output over table counts around the warp's 32 and the row's 8, equally long
strings, empty strings, large buckets, colliding hashed keys, tables sorted in one
block and by radix passes, and a first capacity that is too small."""
import numpy as np
import pytest

import oracle
from paper_1702_00093_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda:0"


@pytest.fixture(scope="module")
def ej():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_00093_gb300 import build
    build.build()
    oracle.build()
    from paper_1702_00093_gb300 import embedjoin
    return embedjoin


def _set(kind, n):
    rng = np.random.default_rng(11 + n)
    lut = np.frombuffer(synth.PROTEIN, np.uint8)
    if kind == "equal":      # one length for all
        lens = np.full(n, 24)
    elif kind == "ragged":   # empty strings among them
        lens = rng.integers(0, 60, size=n)
    else:                    # "long": few lengths, far apart and close together
        lens = rng.choice([30, 31, 32, 70, 71], size=n)
    base = rng.integers(0, 25, size=80)
    strs = []
    for ln in lens:
        s = base[:ln].copy()
        for _ in range(int(rng.integers(0, 6))):
            if ln:
                s[rng.integers(0, ln)] = rng.integers(0, 25)
        strs.append(lut[s].tobytes())
    return synth.pack(strs, synth.PROTEIN)


@pytest.mark.parametrize("r,m", [(1, 1), (2, 4), (3, 11), (4, 16), (5, 13)])
@pytest.mark.parametrize("kind", ["equal", "ragged", "long"])
@pytest.mark.parametrize("P", [0, 13])
def test_grouped_equals_hashed_and_sorted(ej, kind, r, m, P):
    ss = _set(kind, 700)
    s = ej.Strings.from_set(ss, DEV)
    p = ej.Params(K=9, r=r, m=m, z=3, seed=6, L=40, alphabet=ss.alphabet)
    got = {}
    for name, sched in (("grouped", dict(mode=3)), ("hashed", dict(mode=2, buckets=1)), ("sorted", dict(mode=2, buckets=2))):
        ctx = ej.Context(0)   # a new context: the first capacity of each
        ctx.set_key_hash(P)
        ctx.set_schedule(**sched)
        pairs, st = ctx.join(s, p, device=DEV)
        got[name] = (st.n_raw_pairs, st.n_candidates, st.n_out, st.band_cells, pairs.cpu().numpy().view(np.uint64))
        if name != "sorted":
            got[name + "_bucket"] = st.max_bucket
        ctx.close()
    assert got["grouped"][1] > 0
    for other in ("hashed", "sorted"):
        assert got["grouped"][:4] == got[other][:4], other
        assert np.array_equal(got["grouped"][4], got[other][4])
    assert got["grouped_bucket"] == got["hashed_bucket"]


@pytest.mark.parametrize("n", [24576, 24577])
def test_grouped_tables_sorted_in_a_block_and_by_radix(ej, n):
    ss = synth.protein_like(5, n, median=60, sigma_ln=0.3, lo=20, hi=120)
    s = ej.Strings.from_set(ss, DEV)
    p = ej.Params(K=6, r=2, m=5, z=6, seed=6, L=80, alphabet=ss.alphabet)
    out = {}
    for mode in (3, 2):
        ctx = ej.Context(0)
        ctx.set_schedule(mode=mode)
        pairs, st = ctx.join(s, p, device=DEV, capacity=1 << 20)
        out[mode] = (st.n_raw_pairs, st.n_candidates, pairs.cpu().numpy())
        ctx.close()
    assert out[3][:2] == out[2][:2] and out[3][1] > 0
    assert np.array_equal(out[3][2], out[2][2])


def test_grouped_batch_replays_and_tunes(ej):
    """A graph of grouped joins (their tables are sorted inside it) gives each
    join's pairs, also when the choices are tuned first."""
    ss = synth.protein_like(9, 1500, median=120, sigma_ln=0.4, lo=30, hi=400)
    stream = torch.cuda.Stream()
    ctx = ej.Context(0)
    try:
        with torch.cuda.stream(stream):
            s = ej.Strings.from_set(ss, DEV)
            ps = [ej.Params(K=K, r=3, m=5, z=z, seed=2, L=240, alphabet=ss.alphabet) for K, z in ((12, 5), (20, 4))]
            for autotune in (False, True):
                b = ctx.batch(s, ps, autotune=autotune, stream=stream)
                for _ in range(2):
                    b.run(stream)
                    for i, q in enumerate(ps):
                        got, st = b.result(i, device=DEV, stream=stream)
                        ref = oracle.join(ss.data, ss.offsets, ss.alphabet, K=q.K, r=q.r, m=q.m, z=q.z, seed=q.seed, L=q.L)
                        assert st.n_candidates == ref.n_candidates
                        assert np.array_equal(got.cpu().numpy().view(np.uint64), ref.pairs)
                b.close()
    finally:
        ctx.close()
