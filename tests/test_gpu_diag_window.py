"""The diagonal-window verifiers at the edges of their windows: thresholds on both
sides of every 32-diagonal step, strings whose halves end on, just before and just
after a multiple of 32 columns, alphabets of one, four and many symbols. Every
distance is an integer, so the comparison with the oracle is exact."""
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


@pytest.fixture(scope="module")
def ctx(ej):
    c = ej.Context(0)
    yield c
    c.close()


def _edge_set(rng, K, alphabet):
    """Strings whose lengths straddle multiples of 32 and 64 (and very short ones),
    each with copies at 0 .. 2K edits."""
    sigma = len(alphabet)
    lut = np.frombuffer(alphabet, np.uint8)
    strs = []
    for length in (1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 256, 2 * K + 1, 4 * K + 31, 4 * K + 64):
        base = rng.integers(0, sigma, size=max(1, length)).astype(np.uint8)
        strs.append(base)
        for edits in (0, K // 2, K, K + 3, 2 * K):
            strs.append(synth.mutate(rng, base, min(edits, 4 * base.shape[0]), sigma) if sigma > 1 else
                        base[:max(1, base.shape[0] - edits)])
    strs = [s for s in strs if s.shape[0] > 0]
    return synth.pack([lut[s].tobytes() for s in strs], alphabet)


@pytest.mark.parametrize("alphabet", [b"A", b"ACGT", synth.TEXT], ids=["one", "dna", "text"])
@pytest.mark.parametrize("K", [0, 1, 30, 31, 32, 63, 64, 95, 159, 160, 223, 255, 256, 287, 319, 351])
def test_every_window_width_is_exact(ej, ctx, K, alphabet):
    rng = np.random.default_rng(7000 + K)
    ss = _edge_set(rng, K, alphabet)
    p = dict(K=K, r=2, m=4, z=1, seed=4, L=16)
    params = ej.Params(alphabet=alphabet, **p)
    ref = oracle.join(ss.data, ss.offsets, alphabet, **p)
    assert len(ref.pairs) > 0
    s = ej.Strings.from_set(ss, DEV)
    try:
        for mode in (1, 3, 0):
            ctx.set_schedule(mode)
            pairs, st = ctx.join(s, params, device=DEV)
            assert st.n_candidates == ref.n_candidates
            assert np.array_equal(pairs.cpu().numpy().view(np.uint64), ref.pairs), mode
    finally:
        ctx.set_schedule()


def test_search_at_wide_thresholds(ej, ctx):
    """Thresholds beyond the two-lane join verifiers (up to 767 in the persistent
    verifier, wider ones in the grouped one), every query with its own."""
    rng = np.random.default_rng(77)
    lut = np.frombuffer(b"ACGT", np.uint8)
    base = [rng.integers(0, 4, size=int(rng.integers(1500, 2600))).astype(np.uint8) for _ in range(12)]
    idx = synth.pack([lut[b].tobytes() for b in base], b"ACGT")
    Ks = np.array([352, 383, 384, 511, 512, 700, 767, 768, 40, 0], dtype=np.int32)
    qs = [lut[synth.mutate(rng, base[i % 12], int(Ks[i]) + (-20 if i % 2 else 20), 4)].tobytes() for i in range(len(Ks))]
    prm = dict(r=2, m=4, z=1, L=16, seed=2)
    index = ej.Index(ctx, ej.Strings.from_set(idx, DEV), ej.Params(K=0, alphabet=b"ACGT", **prm))
    try:
        got = index.search(qs, Ks)
    finally:
        index.close()
    n = idx.n
    both = synth.pack([idx.get(i) for i in range(n)] + qs, b"ACGT")
    emb, we = oracle.embed(both.data, both.offsets, b"ACGT", prm["r"], prm["L"], prm["seed"])
    keys = oracle.sign(emb, we, oracle.positions(prm["seed"], prm["r"], prm["m"], prm["z"], prm["L"]), 4)
    lens = both.lengths()
    want = []
    for q in range(len(qs)):
        hit = (keys[:, :n] == keys[:, n + q][:, None]).any(axis=0) & (np.abs(lens[:n] - lens[n + q]) <= Ks[q])
        cand = np.nonzero(hit)[0]
        pairs = np.array([(int(i) << 32) | (n + q) for i in cand], dtype=np.uint64)
        ok = oracle.verify(both.data, both.offsets, pairs, int(Ks[q])) == 1 if len(pairs) else np.zeros(0, bool)
        want += [(q << 32) | int(i) for i in cand[ok]]
    assert len(want) > 0
    assert np.array_equal(got, np.array(sorted(want), dtype=np.uint64))
