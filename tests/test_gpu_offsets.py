"""Offsets that are no offsets (decreasing, up and down, beyond the bytes, not from 0):
every call reports EJ_ERR_INVALID_ARG, also where single strings look valid and their
lengths together exceed the bytes, and the context then answers valid input as
before; the same for offsets rewritten between a batch's replays."""
import numpy as np
import pytest

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
    from paper_1702_00093_gb300 import embedjoin
    return embedjoin


def _set(alphabet, n):
    """Pairs of equal strings of 40 to 79 symbols."""
    rng = np.random.default_rng(n)
    lut = np.frombuffer(alphabet, np.uint8)
    strs = []
    for _ in range(n // 2):
        strs += [lut[rng.integers(0, len(alphabet), size=int(rng.integers(40, 80)))].tobytes()] * 2
    return synth.pack(strs, alphabet)


def _malformed(offs):
    """Each with the original's last entry, so that the byte array is the same."""
    total, n = int(offs[-1]), len(offs) - 1
    up_down = np.zeros_like(offs)
    up_down[1::2] = total          # 0, T, 0, T, ...
    up_down[-1] = total
    swapped = offs.copy()
    swapped[[n // 3, n // 2]] = offs[[n // 2, n // 3]]
    below, late, beyond = offs.copy(), offs.copy(), offs.copy()
    below[n // 2] = -1
    late[0] = 1
    beyond[n // 2] = total + 1
    return dict(up_down=up_down, swapped=swapped, below=below, late=late, beyond=beyond)


@pytest.mark.parametrize("n", [301, 20001])   # one-launch and three-launch scans of the chunk counts
@pytest.mark.parametrize("alphabet", [b"ACGT", synth.PROTEIN], ids=["dna", "protein"])
def test_calls_report_malformed_offsets(ej, alphabet, n):
    ss = _set(alphabet, n)
    p = ej.Params(K=2, r=2, m=3, z=8, L=120, seed=4, alphabet=alphabet)
    data, offs = torch.from_numpy(ss.data).to(DEV), torch.from_numpy(ss.offsets).to(DEV)
    good = ej.Strings(data, offs)
    one = torch.ones(1, dtype=torch.int64, device=DEV)
    ctx = ej.Context(0)
    try:
        want, _ = ctx.join(good, p, device=DEV)
        assert len(want) >= n // 2
        for kind, bad in _malformed(ss.offsets).items():
            for s in (ej.Strings(data, torch.from_numpy(bad).to(DEV)), ej.Strings(ss.data, bad)):
                for call in (lambda: ctx.plan(s, p), lambda: ctx.join(s, p, device=DEV)):
                    with pytest.raises(ej.EJError) as e:
                        call()
                    assert e.value.status == ej.EJ_ERR_INVALID_ARG, kind
            with pytest.raises(ej.EJError) as e:
                ej.verify_noalloc(ej.Strings(data, torch.from_numpy(bad).to(DEV)), p, one, torch.empty_like(one))
            assert e.value.status == ej.EJ_ERR_INVALID_ARG, kind
        got, _ = ctx.join(good, p, device=DEV)
        assert torch.equal(got, want)
    finally:
        ctx.close()


@pytest.mark.parametrize("mode", [1, 2, 3])
@pytest.mark.parametrize("alphabet", [b"ACGT", synth.PROTEIN], ids=["dna", "protein"])
def test_batch_replays_report_malformed_offsets(ej, alphabet, mode):
    ss = _set(alphabet, 301)
    p = ej.Params(K=2, r=2, m=3, z=8, L=120, seed=4, alphabet=alphabet)
    ctx, stream = ej.Context(0), torch.cuda.Stream()
    try:
        ctx.set_schedule(mode=mode)
        with torch.cuda.stream(stream):
            s = ej.Strings.from_set(ss, DEV)
            b = ctx.batch(s, [p], stream=stream)
            b.run(stream)
            want, _ = b.result(0, device=DEV, stream=stream)
            assert len(want) >= 150
            for kind in ("swapped", "below", "late", "beyond"):
                s.offsets.copy_(torch.from_numpy(_malformed(ss.offsets)[kind]))
                b.run(stream)
                with pytest.raises(ej.EJError) as e:
                    b.result(0, device=DEV, stream=stream)
                assert e.value.status == ej.EJ_ERR_INVALID_ARG, kind
            s.offsets.copy_(torch.from_numpy(ss.offsets))
            b.run(stream)
            got, _ = b.result(0, device=DEV, stream=stream)
            assert torch.equal(got, want)
            b.close()
    finally:
        ctx.close()


@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("alphabet", [b"ACGT", synth.PROTEIN], ids=["dna", "protein"])
def test_batch_replay_with_a_longer_string(ej, alphabet, lanes):
    """The verifier of four and more lanes per pair sizes its match masks for the
    planned longest string; a replay with a longer one reports it."""
    ss = _set(alphabet, 60)
    p = ej.Params(K=30, r=2, m=3, z=4, L=120, seed=4, alphabet=alphabet)
    ctx, stream = ej.Context(0), torch.cuda.Stream()
    try:
        ctx.set_schedule(mode=2)
        ctx.set_verify_config(lanes, 2 if lanes == 2 else 1)
        with torch.cuda.stream(stream):
            s = ej.Strings.from_set(ss, DEV)
            b = ctx.batch(s, [p], stream=stream)
            b.run(stream)
            want, _ = b.result(0, device=DEV, stream=stream)
            assert len(want) >= 30
            merged = ss.offsets.copy()
            merged[1:40] = merged[40]      # string 0 takes the bytes of the 39 after it
            s.offsets.copy_(torch.from_numpy(merged))
            b.run(stream)
            with pytest.raises(ej.EJError) as e:
                b.result(0, device=DEV, stream=stream)
            assert e.value.status == ej.EJ_ERR_INVALID_ARG
            s.offsets.copy_(torch.from_numpy(ss.offsets))
            b.run(stream)
            got, _ = b.result(0, device=DEV, stream=stream)
            assert torch.equal(got, want)
            b.close()
    finally:
        ctx.close()
