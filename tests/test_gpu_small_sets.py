"""Small sets: outputs on both sides of every size at which the one-block output
sort changes its records per thread (and of its largest), and keys of sets whose
walks are spread over more or fewer blocks."""
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


@pytest.mark.parametrize("same", [2, 45, 46, 64, 65, 91, 92, 128, 129])
@pytest.mark.parametrize("others", [0, 300])
def test_outputs_of_every_sort_size(ej, ctx, same, others):
    """`same` equal strings among unrelated ones: same (same - 1) / 2 output pairs
    (1, 990, 1035, 2016, 2080, 4095, 4186, 8128, 8256), sorted."""
    rng = np.random.default_rng(same)
    lut = np.frombuffer(b"ACGT", np.uint8)
    base = lut[rng.integers(0, 4, size=60)].tobytes()
    strs = [base] * same + [lut[rng.integers(0, 4, size=60)].tobytes() for _ in range(others)]
    order = rng.permutation(len(strs))
    ss = synth.pack([strs[i] for i in order], b"ACGT")
    ids = np.sort(np.nonzero(order < same)[0]).astype(np.uint64)
    i, j = np.triu_indices(same, 1)
    want = (ids[i] << np.uint64(32)) | ids[j]
    p = ej.Params(K=2, r=2, m=4, z=20, seed=1, alphabet=b"ACGT")
    s = ej.Strings.from_set(ss, DEV)
    pairs, _ = ctx.join(s, p, device=DEV)
    assert np.array_equal(pairs.cpu().numpy().view(np.uint64), want)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        b = ctx.batch(s, [p], stream=stream)
        b.run(stream)
        got, _ = b.result(0, device=DEV, stream=stream)
        assert np.array_equal(got.cpu().numpy().view(np.uint64), want)
        b.close()


@pytest.mark.parametrize("alphabet,L", [(b"ACGT", 120), (synth.PROTEIN, 200), (synth.TEXT, 2500)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 700, 2433])
def test_keys_of_spread_walks(ej, ctx, alphabet, L, n):
    rng = np.random.default_rng(n)
    lut = np.frombuffer(alphabet, np.uint8)
    ss = synth.pack([lut[rng.integers(0, len(alphabet), size=int(rng.integers(0, 130)))].tobytes() for _ in range(n)],
                    alphabet)
    prm = dict(r=7, m=5, z=6, L=L, seed=9)
    keys = torch.zeros(prm["r"] * prm["m"] * n, dtype=torch.int64, device=DEV)
    ctx.embed_sign(ej.Strings.from_set(ss, DEV), ej.Params(K=1, out_len=L, alphabet=alphabet, **prm), keys)
    torch.cuda.synchronize()
    want = oracle.keys(ss.data, ss.offsets, alphabet, prm["r"], prm["m"], prm["z"], prm["L"], prm["seed"])
    assert np.array_equal(keys.cpu().numpy().view(np.uint64).reshape(want.shape), want)
