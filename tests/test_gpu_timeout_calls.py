"""Every call whose verification runs on the persistent verifier reports that its loop
bound ran out, and answers exactly with the default bound again."""
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


@pytest.mark.parametrize("call", ["verify", "plus", "join", "grouped"])
def test_loop_bound_reaches_the_call(ej, call):
    ss = synth.dna_clusters(47, 6, 5, 900, 1000, edits_mean=3.0)
    kw = dict(K=20, r=3, m=6, z=8, seed=3, L=900)
    s, p = ej.Strings.from_set(ss, DEV), ej.Params(alphabet=ss.alphabet, **kw)
    if call == "plus":
        ref = oracle.join_plus(ss.data, ss.offsets, ss.alphabet, delta=12, T=1, **kw).pairs
    elif call == "grouped":
        ref, _ = oracle.join_grouped(ss.data, ss.offsets, ss.alphabet, **kw)
    else:
        ref = oracle.join(ss.data, ss.offsets, ss.alphabet, **kw).pairs
    assert len(ref) > 0
    c = ej.Context(0)

    def run():
        if call == "verify":
            cand = torch.from_numpy(ref.view(np.int64)).to(DEV)
            out = torch.zeros_like(cand)
            return out[:c.verify(s, p, cand, out)]
        if call == "plus":
            return c.join_plus(s, p, 12, 1, device=DEV)[0]
        return (c.join if call == "join" else c.join_grouped)(s, p, device=DEV)[0]

    try:
        c.set_loop_bound(1)   # 64 columns of halves of about 480
        with pytest.raises(ej.EJError) as e:
            run()
        assert e.value.status == ej.EJ_ERR_TIMEOUT
        c.set_loop_bound(0)
        assert np.array_equal(run().cpu().numpy().view(np.uint64), ref)
    finally:
        c.close()
