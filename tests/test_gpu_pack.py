"""Packing by byte permutation (alphabets of at most four symbols that three bits
tell apart) and by lookup: the keys, which read every code up to L, equal the
oracle's for alphabets of one to five symbols, also such as no three bits separate,
at every start alignment; and a byte outside the alphabet is reported wherever it
stands, also when its three bits are those of a symbol."""
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


@pytest.mark.parametrize("alphabet", [b"A", b"AT", b"GCA", b"ACGT", bytes([0, 1, 64, 65]), bytes([255, 0, 7]), b"ACGTN"])
@pytest.mark.parametrize("shift", [0, 1, 6, 15])
def test_codes_at_every_alignment(ej, ctx, alphabet, shift):
    rng = np.random.default_rng(17 + shift)
    lut = np.frombuffer(alphabet, np.uint8)
    lens = np.concatenate([np.arange(0, 70), [127, 128, 129, 511, 512, 513, 1040]])
    strs = [lut[rng.integers(0, len(alphabet), size=int(n))].tobytes() for n in rng.permutation(lens)]
    ss = synth.pack(strs, alphabet)
    big = torch.full((len(ss.data) + 32,), 3, dtype=torch.uint8, device=DEV)   # other bytes around the array
    big[shift:shift + len(ss.data)] = torch.from_numpy(ss.data).to(DEV)
    s = ej.Strings(big[shift:shift + len(ss.data)], torch.from_numpy(ss.offsets).to(DEV))
    p = dict(r=2, m=6, z=8, L=1500, seed=5)
    params = ej.Params(K=3, alphabet=alphabet, **p)
    keys = torch.zeros(p["r"] * p["m"] * ss.n, dtype=torch.int64, device=DEV)
    ctx.embed_sign(s, params, keys)
    torch.cuda.synchronize()
    want = oracle.keys(ss.data, ss.offsets, alphabet, p["r"], p["m"], p["z"], p["L"], p["seed"])
    assert np.array_equal(keys.cpu().numpy().view(np.uint64).reshape(want.shape), want)


@pytest.mark.parametrize("alphabet,wrong", [(b"ACGT", b"E"), (b"ACGT", b"N"), (b"ACGT", b"a"), (b"AT", b"C"),
                                            (bytes([0, 1, 64, 65]), bytes([2])), (synth.TEXT, b"~")])
def test_foreign_bytes_are_reported(ej, ctx, alphabet, wrong):
    lut = np.frombuffer(alphabet, np.uint8)
    rng = np.random.default_rng(3)
    ss = synth.pack([lut[rng.integers(0, len(alphabet), size=n)].tobytes() for n in (40, 7, 96, 33)], alphabet)
    params = ej.Params(K=1, r=1, m=1, z=1, alphabet=alphabet)
    for at in (0, 1, 15, 16, 39, 40, 46, 47, 100, 142, 143, len(ss.data) - 1):
        data = ss.data.copy()
        data[at] = wrong[0]
        s = ej.Strings(torch.from_numpy(data).to(DEV), torch.from_numpy(ss.offsets).to(DEV))
        with pytest.raises(ej.EJError) as e:
            ctx.plan(s, params)
        assert e.value.status == ej.EJ_ERR_INVALID_ARG
    ctx.plan(ej.Strings.from_set(ss, DEV), params)
