"""A two-lane tiling asked for is used by joins of short strings of at most four
symbols: with a loop bound of one pass the persistent verifier, which mode 0 takes
there alone or after the shared-string one, runs out, and the tiling asked for, which
has no queue, does not."""
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


@pytest.mark.parametrize("z", [14, 2], ids=["sparse", "dense"])
def test_join_takes_the_tiling_asked_for(ej, z):
    ss = synth.dna_clusters(43, 12, 5, 480, 520, edits_mean=2.0)
    kw = dict(K=6, r=3, m=5, z=z, seed=2, L=600)
    ref = oracle.join(ss.data, ss.offsets, ss.alphabet, **kw)
    assert len(ref.pairs) > 0
    s, p = ej.Strings.from_set(ss, DEV), ej.Params(alphabet=ss.alphabet, **kw)
    c = ej.Context(0)
    try:
        c.set_loop_bound(1)   # 64 columns of halves of about 250
        with pytest.raises(ej.EJError) as e:
            c.join(s, p, device=DEV)
        assert e.value.status == ej.EJ_ERR_TIMEOUT
        for V in (2, 3):
            c.set_verify_config(2, V, 0)
            pairs, st = c.join(s, p, device=DEV)
            assert st.n_candidates == ref.n_candidates
            assert np.array_equal(pairs.cpu().numpy().view(np.uint64), ref.pairs)
        c.set_verify_config(0, 0, 0)
        c.set_loop_bound(0)
        pairs, _ = c.join(s, p, device=DEV)
        assert np.array_equal(pairs.cpu().numpy().view(np.uint64), ref.pairs)
    finally:
        c.close()
