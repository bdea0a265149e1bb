"""Searches that share an index keep their scratch apart: calls of different sizes in
turn, calls from several threads at once, and calls after a rejected one all give
the pairs of a fresh index."""
import threading

import numpy as np
import pytest

from paper_1702_00093_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda:0"
PRM = dict(r=5, m=6, z=8, L=1000, seed=1)


@pytest.fixture(scope="module")
def ej():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_00093_gb300 import build
    build.build()
    from paper_1702_00093_gb300 import embedjoin
    return embedjoin


def test_searches_share_an_index(ej):
    idx = synth.serving_index(3000, seed=31)
    qs, ks = synth.serving_queries(idx, 300, seed=32)
    parts = [(qs[a:b], ks[a:b]) for a, b in ((0, 1), (1, 200), (200, 203), (203, 300), (0, 300))]
    strings = ej.Strings.from_set(idx, DEV)

    def fresh(part):
        ctx = ej.Context(0)
        index = ej.Index(ctx, strings, ej.Params(K=0, alphabet=idx.alphabet, **PRM))
        got = index.search(part[0], part[1])
        index.close()
        ctx.close()
        return got

    want = [fresh(p) for p in parts]
    assert sum(len(w) for w in want) > 0
    owner = ej.Context(0)
    index = ej.Index(owner, strings, ej.Params(K=0, alphabet=idx.alphabet, **PRM))
    for _ in range(2):
        for p, w in zip(parts, want):
            assert np.array_equal(index.search(p[0], p[1]), w)
    with pytest.raises(ej.EJError) as e:
        index.search([b"ACGN"], 3)
    assert e.value.status == ej.EJ_ERR_INVALID_ARG
    assert np.array_equal(index.search(parts[0][0], parts[0][1]), want[0])
    # four threads, each with its own context, on one index
    bad = []

    def work(k):
        torch.cuda.set_device(0)
        ctx = ej.Context(0)
        mine = ej.Index.__new__(ej.Index)   # the same index through this thread's context
        mine._ctx, mine._h, mine.n = ctx, index._h, index.n
        for r in range(6):
            p = (k + r) % len(parts)
            if not np.array_equal(mine.search(parts[p][0], parts[p][1]), want[p]):
                bad.append((k, r))
        mine._h = None
        ctx.close()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    index.close()
    owner.close()
