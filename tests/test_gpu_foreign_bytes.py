"""Bytes outside the alphabet where the strings are walked and verified before the
host reads the error word (a search, a batch's replay): the call reports
EJ_ERR_INVALID_ARG, every code that a kernel sees belongs to the alphabet, and the
same index and batch then answer valid input as before."""
import numpy as np
import pytest

from paper_1702_00093_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda:0"
ALPHABETS = [(synth.PROTEIN, b"J"), (synth.TEXT, b"~"), (b"ACGTN", bytes([255])),
             (b"ACGT", b"N"), (bytes([0, 1, 64]), bytes([2])), (bytes([0, 64]), bytes([1]))]   # packed in 2 bits


@pytest.fixture(scope="module")
def ej():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_00093_gb300 import build
    build.build()
    from paper_1702_00093_gb300 import embedjoin
    return embedjoin


def _set(alphabet):
    """Ten clusters of four similar strings of 90 to 140 symbols."""
    rng = np.random.default_rng(23)
    lut = np.frombuffer(alphabet, np.uint8)
    strs = []
    for _ in range(10):
        base = rng.integers(0, len(alphabet), size=int(rng.integers(90, 141))).astype(np.uint8)
        strs += [lut[synth.mutate(rng, base, int(e), len(alphabet))].tobytes() for e in (0, 1, 2, 4)]
    return synth.pack(strs, alphabet)


def _ids(v):
    return [f"{len(a)}" for a, _ in v]


@pytest.mark.parametrize("L", [200, 1500])   # walk tables of either kind
@pytest.mark.parametrize("alphabet,wrong", ALPHABETS, ids=_ids(ALPHABETS))
def test_search_reports_foreign_bytes(ej, alphabet, wrong, L):
    ss = _set(alphabet)
    ctx = ej.Context(0)
    index = ej.Index(ctx, ej.Strings.from_set(ss, DEV), ej.Params(K=0, r=3, m=4, z=3, L=L, out_len=L, seed=2, alphabet=alphabet))
    try:
        good = [ss.get(i) for i in range(0, ss.n, 4)]
        want = index.search(good, 6)
        assert len(want) >= len(good)   # each finds itself
        for at in (0, 1, 15, 16, 40, 88):
            bad = good[3][:at] + wrong + good[3][at + 1:]
            with pytest.raises(ej.EJError) as e:
                index.search(good[:3] + [bad] + good[4:], 6)
            assert e.value.status == ej.EJ_ERR_INVALID_ARG
        with pytest.raises(ej.EJError) as e:
            index.search([wrong * 120], 6)
        assert e.value.status == ej.EJ_ERR_INVALID_ARG
        assert np.array_equal(index.search(good, 6), want)
    finally:
        index.close()
        ctx.close()


@pytest.mark.parametrize("mode", [1, 2, 3])
@pytest.mark.parametrize("alphabet,wrong", ALPHABETS, ids=_ids(ALPHABETS))
def test_batch_replay_reports_foreign_bytes(ej, alphabet, wrong, mode):
    ss = _set(alphabet)
    ctx, stream = ej.Context(0), torch.cuda.Stream()
    try:
        ctx.set_schedule(mode=mode)
        with torch.cuda.stream(stream):
            s = ej.Strings.from_set(ss, DEV)
            p = ej.Params(K=6, r=3, m=4, z=3, L=200, seed=2, alphabet=alphabet)
            want, _ = ctx.join(s, p, device=DEV, stream=stream)
            assert len(want) > 0
            b = ctx.batch(s, [p], stream=stream)
            for at in (0, 17, len(ss.data) // 2, len(ss.data) - 1):
                keep = s.data[at].clone()
                s.data[at] = wrong[0]
                b.run(stream)
                with pytest.raises(ej.EJError) as e:
                    b.result(0, device=DEV, stream=stream)
                assert e.value.status == ej.EJ_ERR_INVALID_ARG
                s.data[at] = keep
            b.run(stream)
            got, _ = b.result(0, device=DEV, stream=stream)
            assert torch.equal(got, want)
            b.close()
    finally:
        ctx.close()
