"""The logits window after a layer selection: the wide LM head and the
hidden-state DP of a bf16 model write no logits, so the window keeps those of
the pass before."""
import numpy as np
import pytest

from helpers import need_gpu
from test_gpu_wide_edges import shape_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def test_selection_leaves_the_logits():
    from paper_2602_20217_gb300 import knapspec as ks
    from paper_2602_20217_gb300 import synth
    from paper_2602_20217_gb300.model import Model
    shape = shape_of(vocab=2000)
    m = Model(shape, max_seq=256, seed=0)
    m.prefill(synth.prompt_tokens(shape, 40, seed=1))
    m.draft(np.ones(shape.n_sublayers, np.uint8), 7)
    m.verify(None, 7)
    before = m.logits(8)
    m.select_tpt(ks.latency(0, 0.08, 2e-5, 0.05), 8, 10)
    assert np.array_equal(before, m.logits(8))
    m.select_dp(ks.latency(1, units=np.ones(shape.n_sublayers, np.int32)), 8, tau=-2.0, max_states=8, max_rows=16)
    assert np.array_equal(before, m.logits(8))
    m.close()
