"""The verifier that a join over at most four symbols takes by itself: the shared-string
one when chance fills its tasks, the persistent one when a window of many words or
classes leaves them nearly empty. Either counts its own word-columns, which tell the
choice; the pairs are the same."""
import numpy as np
import pytest

from paper_1702_00093_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda:0"


# (length, K, z, tables, the choice): chance = 0.5 tables 600 4^-z against W classes / 3,
# times the root of tables / 152
@pytest.mark.parametrize("length,K,z,r,m,mode", [
    (1000, 250, 5, 4, 5, 1),     # 5.9 against 7.6: the window has 9 words, 7 classes
    (1000, 250, 4, 4, 5, 3),     # 23
    (1000, 60, 5, 2, 7, 3),      # 4.1 against 3.2 (2 words, 16 classes)
    (1000, 60, 6, 5, 8, 1),      # 2.9 against 5.5
    (300, 10, 6, 4, 10, 3),      # 2.9 against 2 (one class)
    (300, 10, 6, 2, 10, 1),      # 1.5
])
def test_choice_of_mode_0(length, K, z, r, m, mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_00093_gb300 import build
    build.build()
    from paper_1702_00093_gb300 import embedjoin as ej
    ss = synth.dna_clusters(4, 60, 10, int(0.9 * length), int(1.1 * length), rate_lo=0.01, rate_hi=0.08)
    s = ej.Strings.from_set(ss, DEV)
    p = ej.Params(K=K, r=r, m=m, z=z, seed=1, L=length, alphabet=ss.alphabet)
    got = {}
    for k in (0, 1, 2, 3):
        ctx = ej.Context(0)
        ctx.set_schedule(mode=k)
        pairs, st = ctx.join(s, p, device=DEV)
        got[k] = (st.n_candidates, st.band_cells, st.verify_word_columns, pairs.cpu().numpy())
        ctx.close()
    assert got[1][2] != got[3][2]
    assert got[0][2] == got[mode][2]
    for k in (0, 1, 3):
        assert got[k][:2] == got[2][:2]
        assert np.array_equal(got[k][3], got[2][3])
