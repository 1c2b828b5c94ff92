"""The hidden-state DP's states in wide passes, state by state against the fp64
oracle, at the edges of their attention: a sequence that is all history (no
cache below the states), a prefix of several key tiles, one and two query
tiles, own keys that do not begin at a tile, states across tile and CTA edges
and longer than a tile, several batches of states, both head sizes.

With tau below every cosine each reachable skipped weight survives, so the
candidates' skipped weights are the subset sums of the units, and a
candidate's state is its layer set run on the history rows: the target's K/V
below them, the state's own K/V among them.  The last layer weighs more than
every state it is evaluated for, so no skip can stand in for a state that its
attention spoils.

Tolerance: the bf16 tolerance of the decoder tests, 2e-2 of a row's largest
entry; acceptances may differ by the rows whose two best logits lie within it."""
import numpy as np
import pytest

from helpers import need_gpu, oracle_model, rel_err
from oracle import decoder as D
from oracle import dp as DP

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def reachable(units, jmax):
    js = {0}
    for u in units:
        js |= {j + u for j in js if j + u <= jmax}
    return sorted(js, reverse=True)


def sequence(m, prompt, gammas):
    """The committed tokens after a prompt and a verify step per draft length."""
    seq = list(prompt) + [m.prefill(prompt)]
    full = np.ones(m.shape.n_sublayers, np.uint8)
    for g in gammas:
        m.draft(full, g)
        a, new = m.verify(None, g)
        assert a == g                       # drafts of the full model
        seq += [int(t) for t in new]
    return seq[:-1]


def run_dp(m, units, max_rows, tau):
    """The DP's candidates and the final states of all skipped weights, [S][r][d]."""
    import torch

    from paper_2602_20217_gb300 import knapspec as ks
    S = int(np.sum(units)) // 2 + 1
    r = min(int(ks.ks_debug_read(m.h, 4, 0, 0, 0, np.zeros(1, np.int32))[0]), max_rows)
    nb = ks.load().ks_dp_scratch_bytes(m.h, S, max_rows)
    scratch = torch.zeros(nb + 256, dtype=torch.uint8, device="cuda")
    off = -scratch.data_ptr() % 256
    lat, _u = ks.latency(1, units=np.asarray(units, np.int32))
    out = ks.ks_select_dp(m.h, lat, m.shape.n_sublayers, tau, 4, S, max_rows, scratch.data_ptr() + off, nb)
    d = m.shape.d_model
    states = scratch[off: off + 4 * S * r * d].view(torch.float32).view(S, r, d).cpu().numpy()
    return out, states, r


def shape_of(hd, L=4, d=512, hq=8, hk=2, ff=1368):
    from paper_2602_20217_gb300.configs import ModelShape
    return ModelShape(f"dp-{hd}-{d}", L, d, hq, hk, hd, ff, 2000, qk_norm=hd == 128, dtype="bf16",
                      rope_theta=500000.0)


# units of 8 sublayers: the first six reach every skipped weight up to 8 / 24
UNITS8 = [1, 2, 1, 1, 2, 1, 9, 9]                # 14 states: 13 evaluated
UNITS24 = [1, 2, 4, 8, 6, 3, 25, 25]             # 38 states: 37 evaluated


@pytest.mark.parametrize("n,gammas,rows,units,hd", [
    (8, [5, 5], 64, UNITS24, 128),               # 37 x 20 rows, no cache below them; two batches
    (8, [5, 5], 64, UNITS24, 64),
    (5, [4, 8, 8], 64, UNITS24, 128),            # 37 x 28
    (8, [15], 64, UNITS8, 128),                  # 13 x 24, two query blocks
    (8, [1], 64, UNITS8, 64),                    # 13 x 10, two query tiles
    (300, [15, 6], 23, UNITS24, 128),            # 37 x 23, prefix of three tiles
    (300, [15, 6], 23, UNITS24, 64),
    (140, [6], 15, UNITS8, 64),                  # 13 x 15, prefix of two tiles
])
def test_states_match_the_oracle(n, gammas, rows, units, hd):
    check(shape_of(hd), n, gammas, rows, units)


def test_states_longer_than_a_key_tile():
    check(shape_of(128), 8, [15] * 8, 130, UNITS8, hist_steps=12)     # 13 x 130, 6 positions below them


def test_predictions_in_several_batches():
    # a narrow model's LM head rows: room for about 570 at a time, 14 x 56 here
    from paper_2602_20217_gb300.configs import ModelShape
    check(ModelShape("dp-narrow", 4, 2048, 1, 1, 64, 8, 300, dtype="bf16"), 8, [15] * 3, 56, UNITS8)


def check(shape, n, gammas, rows, units, hist_steps=5):
    from paper_2602_20217_gb300 import synth
    from paper_2602_20217_gb300.model import Model
    m = Model(shape, max_seq=512, seed=0, hist_steps=hist_steps)
    seq = sequence(m, synth.prompt_tokens(shape, n, seed=1), gammas)
    p = m.position()[0]
    assert p == len(seq)
    (mask, g, tpt, js, alphas, cands), states, r = run_dp(m, units, rows, tau=-2.0)
    assert list(js) == reachable(units, sum(units) // 2)
    cfg, w = oracle_model(shape, seed=0)
    s = D.Session(cfg, w, p + 8, hist_steps=5, hist_init_rows=r)
    s.prefill(seq, chunk=len(seq))
    hist = s.history()
    assert hist.shape[1] == r and s.p == p
    target = D.final_logits(cfg, w, hist[-1])
    for j, cand, alpha in zip(js, cands, alphas):
        assert sum(u for u, x in zip(units, cand) if not x) == j
        x = hist[0]
        for i in range(1, shape.n_sublayers + 1):
            if cand[i - 1]:
                l = (i - 1) // 2
                kv = {l: (s.k[l].copy(), s.v[l].copy())} if i % 2 == 1 else {}
                x = DP.sublayer(s, i, x, p - r, kv)
        assert np.all(np.isfinite(states[j])), j
        assert rel_err(states[j], x) < 2e-2, j
        lg = D.final_logits(cfg, w, x)
        unsure = np.count_nonzero(near_tie(lg) | near_tie(target))
        same = np.count_nonzero(np.argmax(lg, -1) == np.argmax(target, -1))
        assert abs(alpha * r - same) <= unsure + 1e-9, j
    m.close()


def near_tie(logits):
    best = np.sort(logits, axis=-1)
    return best[:, -1] - best[:, -2] < 2e-2 * np.max(np.abs(logits), axis=-1)
