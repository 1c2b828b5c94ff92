"""The sampling filter over rows of one slice and several rounds of slices, with
equal logits at the cut (tests/test_gpu_sampling.py has the rest).

Tolerance on probabilities: the sampling tests' 1e-5 (fp32 sums of at most 64
terms against fp64)."""
import numpy as np
import pytest

from helpers import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("vocab", [5, 70, 16385, 131073, 300001])
def test_filter_over_long_rows_with_ties(vocab):
    """Rows of one to three rounds of the filter's slices; every LM head row
    appears several times, so equal logits straddle the cut: lower ids stay."""
    from oracle import sampling as SP
    from paper_2602_20217_gb300 import knapspec as ks
    from paper_2602_20217_gb300 import synth
    from paper_2602_20217_gb300.configs import ModelShape
    from paper_2602_20217_gb300.model import Model
    shape = ModelShape(f"filter-{vocab}", 1, 64, 1, 1, 64, 64, vocab, dtype="bf16", rope_theta=500000.0)
    w = synth.torch_model_weights(shape, 0)
    w["lm_head"] = w["lm_head"][(synth.np_tokens(77, vocab, max(1, vocab // 7))).astype(np.int64)].contiguous()
    m = Model(shape, max_seq=64, weights=w)
    m.prefill(synth.prompt_tokens(shape, 20, seed=1))
    for k, p in ((1, 1.0), (50, 0.95), (64, 1.0)):
        m.rewind()
        m.draft_sample(np.ones(2, np.uint8), 1, ks.sampling(0.7, k, p, seed=3), 0)
        ids, pr = ks.ks_sample_dists(m.h, "draft", 0, 1)[0]
        ref_ids, ref_pr = SP.filter_distribution(m.logits(1)[0], 0.7, k, p)
        assert abs(len(ids) - len(ref_ids)) <= 1          # the top-p cut may round either way
        n = min(len(ids), len(ref_ids))
        assert np.array_equal(ids[:n], ref_ids[:n])
        if len(ids) == len(ref_ids):
            assert np.max(np.abs(pr.astype(np.float64) - ref_pr)) < 1e-5
    m.close()
