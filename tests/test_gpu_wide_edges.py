"""Edges of the many-row passes that only unusual sizes reach.

* Tiles cut along K (more than 7680 inputs and few tiles): every projection
  kind, whole rounds before the cut tiles, both head sizes; the comparison and
  its tolerance are test_gpu_wide.py's.
* The TPT stage's LM head over cut tiles and in several batches of rows: the
  oracle's acceptances from the GPU's own history, up to the rows whose two
  best logits lie within the bf16 tolerance (2e-2 of the largest)."""
import numpy as np
import pytest

from helpers import need_gpu, oracle_model
from oracle import decoder as D
from oracle import select as S
from test_gpu_dp_states import near_tie, sequence
from test_gpu_wide import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def shape_of(L=2, d=512, hq=8, hk=2, hd=128, ff=1368, vocab=333, qk_norm=False):
    from paper_2602_20217_gb300.configs import ModelShape
    return ModelShape(f"edge-{d}-{ff}-{hq}", L, d, hq, hk, hd, ff, vocab, qk_norm=qk_norm, dtype="bf16",
                      rope_theta=500000.0)


@pytest.mark.parametrize("n,kw", [
    (300, dict(ff=8264)),                                           # W_down, ragged K
    (100, dict(ff=8264)),
    (300, dict(hq=64, hk=4)),                                       # W_o
    (300, dict(d=8192, hq=4, hk=2, ff=264, qk_norm=True)),          # QKV and gate/up
    (300, dict(d=8192, hq=4, hk=2, hd=64, ff=264, qk_norm=True)),   # (without the norm the scores have a spread of 3
                                                                    # and bf16 rounding alone makes 2.2e-2 of the logits)
    (2048, dict(L=1, d=2560, hq=2, hk=1, ff=8264)),                 # 80 tiles of W_down: 76 whole, 4 cut
])
def test_cut_tiles(n, kw):
    check(shape_of(**kw), n)


@pytest.mark.parametrize("shape_kw,gammas,K", [
    (dict(d=8192, hq=4, hk=2, ff=264, vocab=700), [5, 5], 8),       # cut tiles of the LM head
    (dict(d=2048, hq=1, hk=1, hd=64, ff=8, vocab=300), [15] * 3, 16),   # 17 x 56 rows, room for about 570
])
def test_tpt_predictions(shape_kw, gammas, K):
    check_tpt(shape_of(**shape_kw), gammas, K)


def check_tpt(shape, gammas, K):
    from paper_2602_20217_gb300 import knapspec as ks
    from paper_2602_20217_gb300 import synth
    from paper_2602_20217_gb300.model import Model
    cfg, w = oracle_model(shape, seed=0)
    m = Model(shape, max_seq=256, seed=0)
    sequence(m, synth.prompt_tokens(shape, 40, seed=1), gammas)
    mask, g, tpt, alphas, cand = m.select_tpt(ks.latency(0, 0.08, 2e-5, 0.05), K, 10)
    hist = m.history().astype(np.float64)
    r = hist.shape[1]
    target = D.final_logits(cfg, w, hist[-1])
    for j in range(K):
        lg = D.final_logits(cfg, w, S.draft_states(hist, cand[j]))
        unsure = np.count_nonzero(near_tie(lg) | near_tie(target))
        same = np.count_nonzero(np.argmax(lg, -1) == np.argmax(target, -1))
        assert abs(alphas[j] * r - same) <= unsure + 1e-9, j
    m.close()
