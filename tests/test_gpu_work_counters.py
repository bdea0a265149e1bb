"""The persistent verifier's counters belong to the pairs: whatever slots and warps run
them, in whatever order their slots refill, each pair is rejected after the same
columns."""
import numpy as np
import pytest

from paper_1702_00093_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda:0"


@pytest.mark.parametrize("kind", ["text", "dna"])
def test_word_columns_do_not_depend_on_the_refills(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_00093_gb300 import build
    build.build()
    from paper_1702_00093_gb300 import embedjoin as ej
    if kind == "text":
        ss = synth.text_like(8, 2500, len_lo=60, len_hi=700, rate_lo=0.01, rate_hi=0.2)
        p = ej.Params(K=60, r=3, m=4, z=3, seed=1, L=500, alphabet=ss.alphabet)
    else:
        ss = synth.dna_clusters(9, 250, 10, 100, 900, rate_lo=0.01, rate_hi=0.15)
        p = ej.Params(K=40, r=3, m=4, z=4, seed=1, L=400, alphabet=ss.alphabet)
    s = ej.Strings.from_set(ss, DEV)
    ctx = ej.Context(0)
    seen, pairs = set(), None
    try:
        for slots, warps, order in ((16, 1, 4), (16, 1, 4), (16, 4, 4), (8, 1, 2), (3, 1, 3), (1, 2, 4)):
            ctx.set_schedule(mode=1, slots_per_warp=slots, warps_per_subpartition=warps, order=order)
            got, st = ctx.join(s, p, device=DEV, capacity=1 << 18)
            assert st.n_candidates > 2 * 152 * 4 * 16   # every slot refills
            seen.add((st.n_candidates, st.band_cells, st.verify_word_columns))
            pairs = got if pairs is None else pairs
            assert torch.equal(got, pairs)
    finally:
        ctx.close()
    assert len(seen) == 1, seen
