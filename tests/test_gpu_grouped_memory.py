"""The shared-string verifier's buffers: device memory per string of a join with many
classes of the length difference and few candidates, more pairs handed to the
persistent verifier than its list holds, and windows kept from class to class in some
tables and searched anew in the others (more than 160 tables)."""
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


def _u64(t):
    return t.cpu().numpy().view(np.uint64)


def test_memory_per_string(ej):
    """200000 unrelated strings at K = 300 (16 classes): the tasks take about 1.1 KB a
    string, four sorted tables and the strings below 0.7 KB; a full set of tasks per
    class, in every pair buffer, would be 12 KB."""
    n = 200000
    rng = np.random.default_rng(3)
    lens = rng.integers(50, 81, size=n)
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    data = np.frombuffer(synth.PROTEIN, np.uint8)[rng.integers(0, 25, size=int(offs[-1]))]
    s = ej.Strings(torch.from_numpy(data).to(DEV), torch.from_numpy(offs).to(DEV))
    out = torch.zeros(1 << 16, dtype=torch.int64, device=DEV)
    p = ej.Params(K=300, r=2, m=2, z=10, L=60, seed=1, alphabet=synth.PROTEIN)
    small = ej.Context(0)   # what any context and the loaded kernels take
    small.set_schedule(mode=3)
    small.join_into(ej.Strings(s.data, s.offsets[:1001].clone()), p, out)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info(0)[0]
    ctx = ej.Context(0)
    ctx.set_schedule(mode=3)
    _, st = ctx.join_into(s, p, out)
    used = free - torch.cuda.mem_get_info(0)[0]
    ctx.close()
    small.close()
    assert st.n_candidates < 4 * n   # the first capacity was enough
    assert used < 3072 * n, used / n


def test_more_pairs_handed_on_than_the_list_holds(ej):
    """80 clusters of 48 strings: one prefix, one of two tails, lengths in 8 steps of two
    classes, so that every task has at most 6 pairs and hands them on: 90240 pairs,
    and a first capacity of 65536 for 3840 strings."""
    rng = np.random.default_rng(5)
    lut = np.frombuffer(synth.PROTEIN, np.uint8)
    strs = []
    for _ in range(80):
        head = rng.integers(0, 25, size=700)
        tails = rng.integers(0, 25, size=(48, 560))
        for step in range(8):
            for k in range(6):
                tail = tails[0] if k < 3 else tails[6 * step + k]   # three alike, three on their own
                strs.append(lut[np.concatenate([head, tail[:560 - 40 * step]])].tobytes())
    ss = synth.pack(strs, synth.PROTEIN)
    s = ej.Strings.from_set(ss, DEV)
    p = ej.Params(K=300, r=2, m=2, z=12, L=400, seed=1, alphabet=synth.PROTEIN)
    got = {}
    for mode in (3, 2):
        ctx = ej.Context(0)
        ctx.set_schedule(mode=mode)
        pairs, st = ctx.join(s, p, device=DEV, capacity=1 << 17)
        got[mode] = (st.n_candidates, st.band_cells, _u64(pairs))
        ctx.close()
    assert got[3][0] == got[2][0] == 80 * 48 * 47 // 2
    assert got[3][1] == got[2][1]
    assert 0 < len(got[3][2]) < 65536
    assert np.array_equal(got[3][2], got[2][2])
    first = np.array([(i << 32) | j for i in range(48) for j in range(i + 1, 48)], dtype=np.uint64)
    ok = first[oracle.verify_cutoff(ss.data, ss.offsets, first, p.K) == 1]
    assert np.array_equal(got[3][2][: len(ok)], ok)


@pytest.mark.parametrize("r,m", [(5, 32), (7, 23), (12, 20)])   # 160, 161 and 240 tables
def test_windows_of_many_tables(ej, r, m):
    rng = np.random.default_rng(r * m)
    lut = np.frombuffer(synth.PROTEIN, np.uint8)
    base = rng.integers(0, 25, size=170)
    strs = []
    for _ in range(400):
        x = base[: int(rng.integers(60, 171))].copy()
        hit = rng.integers(0, len(x), size=int(rng.integers(0, 30)))
        x[hit] = rng.integers(0, 25, size=len(hit))
        strs.append(lut[x].tobytes())
    ss = synth.pack(strs, synth.PROTEIN)
    s = ej.Strings.from_set(ss, DEV)
    kw = dict(r=r, m=m, z=4, seed=9, L=120)
    for K in (28, 60, 95):   # 8, 16 and 3 classes
        got = {}
        for mode in (3, 2):
            ctx = ej.Context(0)
            ctx.set_schedule(mode=mode)
            pairs, st = ctx.join(s, ej.Params(K=K, alphabet=ss.alphabet, **kw), device=DEV)
            got[mode] = (st.n_raw_pairs, st.n_candidates, st.max_bucket, st.band_cells, _u64(pairs))
            ctx.close()
        ref = oracle.join(ss.data, ss.offsets, ss.alphabet, K=K, **kw)
        assert got[3][:4] == got[2][:4]
        assert got[3][1] == ref.n_candidates > 0
        assert np.array_equal(got[3][4], ref.pairs) and np.array_equal(got[2][4], ref.pairs)


def test_handed_on_pairs_do_not_depend_on_the_capacity(ej):
    """More pairs are handed on than the first capacity has, and fewer than a capacity
    raised by a larger join before: the same pairs take the second verifier."""
    rng = np.random.default_rng(6)
    lut = np.frombuffer(synth.PROTEIN, np.uint8)
    strs = []
    for _ in range(80):
        head, tail = rng.integers(0, 25, size=700), rng.integers(0, 25, size=560)
        for step in range(8):
            for k in range(6):
                end = tail if k < 3 else rng.integers(0, 25, size=560)
                strs.append(lut[np.concatenate([head, end[:560 - 40 * step]])].tobytes())
    s = ej.Strings.from_set(synth.pack(strs, synth.PROTEIN), DEV)
    p = ej.Params(K=300, r=2, m=2, z=12, L=400, seed=1, alphabet=synth.PROTEIN)
    n = 50000
    large = ej.Strings(torch.from_numpy(lut[rng.integers(0, 25, size=140 * n)]).to(DEV),
                       torch.arange(0, 140 * n + 1, 140, dtype=torch.int64, device=DEV))
    got = []
    for larger_first in (False, True):
        ctx = ej.Context(0)
        ctx.set_schedule(mode=3)
        if larger_first:
            ctx.join(large, p, device=DEV)
        pairs, st = ctx.join(s, p, device=DEV, capacity=1 << 17)
        got.append((st.n_candidates, st.band_cells, st.verify_word_columns, _u64(pairs)))
        ctx.close()
    assert got[0][0] == 80 * 48 * 47 // 2   # above the first capacity of 65536
    assert got[0][:3] == got[1][:3]
    assert np.array_equal(got[0][3], got[1][3])


def test_more_pairs_kept_than_the_first_capacity(ej):
    """Clusters of 12 equal strings give 5.5 output pairs a string where the first
    capacity is 4: the first join of a context does no more than the second."""
    n = 24000
    rng = np.random.default_rng(8)
    data = np.frombuffer(synth.PROTEIN, np.uint8)[np.repeat(rng.integers(0, 25, size=(n // 12, 80)), 12, axis=0)]
    s = ej.Strings(torch.from_numpy(data.reshape(-1).copy()).to(DEV),
                   torch.arange(0, 80 * n + 1, 80, dtype=torch.int64, device=DEV))
    p = ej.Params(K=20, r=2, m=2, z=12, L=60, seed=1, alphabet=synth.PROTEIN)
    want = np.array([(12 * c + i) << 32 | (12 * c + j) for c in range(n // 12) for i in range(12)
                     for j in range(i + 1, 12)], dtype=np.uint64)
    ctx = ej.Context(0)
    ctx.set_schedule(mode=3)
    launches = []
    for _ in range(2):
        pairs, st = ctx.join(s, p, device=DEV, capacity=1 << 18)
        assert np.array_equal(_u64(pairs), want)
        launches.append(st.kernel_launches)
    ctx.close()
    assert launches[0] == launches[1]
