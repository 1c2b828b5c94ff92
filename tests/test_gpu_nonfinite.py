"""Non-finite values stay where they belong in the many-row attention: a row
depends on the rows it sees and on nothing else, whatever the others hold.

* A token whose embedding is infinite leaves the prompt's rows before it
  exactly as they are without it.
* K/V rows that an earlier prompt left behind (past the new prompt, in the
  next head's or layer's rows) do not reach a later prompt.
* In the hidden-state DP a state that overflows does not touch the others.

All comparisons are exact: the same rows go through the same operations."""
import numpy as np
import pytest

from helpers import need_gpu
from test_gpu_dp_states import run_dp, sequence

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def shape_of(hd, L=2):
    from paper_2602_20217_gb300.configs import ModelShape
    return ModelShape(f"nonfinite-{hd}", L, 512, 8, 2, hd, 1368, 2000, qk_norm=hd == 128, dtype="bf16",
                      rope_theta=500000.0)


BAD = 7


def setup(shape, max_seq):
    """A model one of whose tokens is infinite, and a prompt source without it."""
    from paper_2602_20217_gb300 import synth
    from paper_2602_20217_gb300.model import Model
    weights = synth.torch_model_weights(shape, 0)
    weights["embed"][BAD] = float("inf")

    def prompt(n, seed):
        t = synth.prompt_tokens(shape, n, seed=seed)
        return np.where(t == BAD, BAD + 1, t).astype(np.int32)

    return Model(shape, max_seq=max_seq, weights=weights), prompt


def cache(m, n):
    return [m.kv(l, 0, n, which) for l in range(m.shape.n_layers) for which in ("k", "v")]


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("n,at", [(200, 150), (300, 129), (300, 256), (700, 300), (2300, 2050)])
def test_rows_before_a_bad_token(hd, n, at):
    m, prompt = setup(shape_of(hd), n + 8)
    t = prompt(n, 1)
    m.prefill(t)
    good = cache(m, n)
    t[at] = BAD
    m.prefill(t)
    for i, (a, b) in enumerate(zip(good, cache(m, n))):
        assert np.array_equal(a[:, :at], b[:, :at])
        if i >= 2:                           # every later row of the second layer sees the bad token
            assert not np.any(np.isfinite(b[:, at:]).all(axis=-1))
    m.close()


@pytest.mark.parametrize("n,max_seq", [(100, 208), (190, 208), (260, 300)])
def test_rows_an_earlier_prompt_left(n, max_seq):
    shape = shape_of(128)
    m, prompt = setup(shape, max_seq)
    t = prompt(n, 2)
    m.prefill(t)
    good, logits = cache(m, n), m.logits(16)
    bad = prompt(max_seq - 1, 3)
    bad[3] = BAD
    m.prefill(bad)
    m.prefill(t)
    assert np.array_equal(logits, m.logits(16))
    assert all(np.array_equal(a, b) for a, b in zip(good, cache(m, n)))
    m.close()


@pytest.mark.parametrize("n,gammas", [(6, [2]), (6, [15, 15, 12])])
def test_a_state_that_overflows(n, gammas):
    """Residual column C holds 10 in every row; the first MLP adds about 1e4 to
    column M, so a state that runs it has column C near 0.02 after the norm,
    one that skips it near 20, and the second layer's value feature 0 = 2e37
    times that overflows in the latter alone.  Nothing reads that feature
    (W_o's columns for it are zero): the others are the states of the model
    without it."""
    from paper_2602_20217_gb300 import synth
    from paper_2602_20217_gb300.model import Model
    shape = shape_of(128)
    C, M, hd, hq, hk, ff = 5, 9, 128, 8, 2, shape.d_ff
    units = [1, 2, 4, 8]                      # every skipped weight is one layer set; 2 and 3 run the overflow
    results = []
    for v in (0.0, 2e37):
        weights = synth.torch_model_weights(shape, 0)
        weights["embed"][:, C] = 10.0
        first, second = weights["layers"]
        first["w_gate_up"][0] = 0.0
        first["w_gate_up"][ff] = 0.0
        first["w_gate_up"][0, C] = first["w_gate_up"][ff, C] = 1.0
        first["w_down"][:, 0] = 0.0
        first["w_down"][M, 0] = 20.0
        second["w_qkv"][(hq + hk) * hd] = 0.0
        second["w_qkv"][(hq + hk) * hd, C] = v
        second["w_o"][:, [h * hd for h in range(hq // hk)]] = 0.0
        m = Model(shape, max_seq=256, weights=weights)
        sequence(m, synth.prompt_tokens(shape, n, seed=1), gammas)
        (mask, g, tpt, js, alphas, cands), states, r = run_dp(m, units, 64, tau=-2.0)
        results.append((list(js), {j: (c, states[j]) for j, c in zip(js, cands)}))
        m.close()
    (js0, clean), (js1, over) = results
    assert js0 == [7, 6, 5, 4, 3, 2, 1, 0]
    assert js1 == [7, 6, 5, 4, 1, 0]
    for j in js1:
        assert np.array_equal(clean[j][0], over[j][0]) and np.array_equal(clean[j][1], over[j][1]), j
