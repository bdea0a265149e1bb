"""The persistent verifier's wide windows (13 to 24 words): thresholds on both sides of
every step, and searches with alphabets near the largest that each window's match
words hold, on an index with a string too long for the verifier of several lanes per
pair. Distances are integers, so the comparison with the oracle is exact."""
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


@pytest.mark.parametrize("alphabet", [b"ACGT", b"ACGTN", bytes(range(60, 95))], ids=["dna", "five", "35"])
@pytest.mark.parametrize("K", [383, 384, 447, 448, 511, 512, 575, 576, 639, 640, 703, 704, 767])
def test_verify_at_every_window_step(ej, ctx, K, alphabet):
    rng = np.random.default_rng(K)
    lut = np.frombuffer(alphabet, np.uint8)
    strs = []
    for length in (K + 1, 1200, 2111):
        base = rng.integers(0, len(alphabet), size=length).astype(np.uint8)
        strs += [lut[base].tobytes()]
        strs += [lut[synth.mutate(rng, base, e, len(alphabet))].tobytes() for e in (3, K - 9, K, K + 25)]
    ss = synth.pack(strs, alphabet)
    pairs = np.array([(i << 32) | j for i in range(ss.n) for j in range(i + 1, ss.n)], dtype=np.uint64)
    want = pairs[oracle.verify(ss.data, ss.offsets, pairs, K) == 1]
    assert 0 < len(want) < len(pairs)
    out = torch.zeros(len(pairs), dtype=torch.int64, device=DEV)
    n = ctx.verify(ej.Strings.from_set(ss, DEV), ej.Params(K=K, r=1, m=1, z=1, L=16, alphabet=alphabet),
                   torch.from_numpy(pairs.view(np.int64)).to(DEV), out)
    assert np.array_equal(np.sort(out[:n].cpu().numpy().view(np.uint64)), want)


# (symbols, thresholds): the largest alphabets that windows of whole 64-bit words held
@pytest.mark.parametrize("sigma,Ks", [(55, (330, 384)), (48, (385, 448)), (44, (449, 512)), (40, (513, 576)),
                                      (36, (577, 640)), (33, (641, 704))])
def test_search_with_large_alphabets(ej, ctx, sigma, Ks):
    rng = np.random.default_rng(sigma)
    alphabet = bytes(range(40, 40 + sigma))
    lut = np.frombuffer(alphabet, np.uint8)
    base = [rng.integers(0, sigma, size=int(ln)).astype(np.uint8) for ln in (1500, 1700, 2100, 2400, 42000)]
    idx = synth.pack([lut[b].tobytes() for b in base], alphabet)
    K = np.array([k for k in Ks for _ in range(3)], dtype=np.int32)
    which = [0, 3, 4, 1, 2, 4]
    edits = [-30, 20, -30, 5, -25, 10]
    qs = [lut[synth.mutate(rng, base[w], int(k) + e, sigma)].tobytes() for w, e, k in zip(which, edits, K)]
    prm = dict(r=2, m=4, z=1, L=16, seed=2)
    index = ej.Index(ctx, ej.Strings.from_set(idx, DEV), ej.Params(K=0, alphabet=alphabet, **prm))
    try:
        got = index.search(qs, K)
    finally:
        index.close()
    n = idx.n
    both = synth.pack([idx.get(i) for i in range(n)] + qs, alphabet)
    emb, we = oracle.embed(both.data, both.offsets, alphabet, prm["r"], prm["L"], prm["seed"])
    keys = oracle.sign(emb, we, oracle.positions(prm["seed"], prm["r"], prm["m"], prm["z"], prm["L"]), sigma)
    lens = both.lengths()
    want = []
    for q in range(len(qs)):
        hit = (keys[:, :n] == keys[:, n + q][:, None]).any(axis=0) & (np.abs(lens[:n] - lens[n + q]) <= K[q])
        cand = np.nonzero(hit)[0]
        pairs = np.array([(int(i) << 32) | (n + q) for i in cand], dtype=np.uint64)
        ok = oracle.verify_cutoff(both.data, both.offsets, pairs, int(K[q])) == 1 if len(pairs) else np.zeros(0, bool)
        want += [(q << 32) | int(i) for i in cand[ok]]
    assert len(want) > 0
    assert np.array_equal(got, np.array(sorted(want), dtype=np.uint64))
