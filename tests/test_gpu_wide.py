"""Prompt processing in wide chunks (tensor-core GEMMs and attention over many
rows) against the fp64 oracle at the sizes where it can go wrong: around the
shortest prompt that takes the path (33 tokens at 16 rows per pass), the edges
of the 128- and 256-row tiles, several chunks, ragged d_ff / vocabulary
/ d_model, both head sizes, few and many query heads per KV head.

Tolerance: the bf16 tolerance of the decoder tests (2e-2 of a row's largest
logit) for the logits, and 2e-2 of a layer's largest entry for K and V, whose
own rounding to bf16 is 2^-9 of an entry."""
import numpy as np
import pytest

from helpers import need_gpu, oracle_model, rel_err
from oracle import decoder as D

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def shape_of(hd=128, qk_norm=True, hq=8, hk=2, d=512, ff=1368, vocab=2000, L=2):
    from paper_2602_20217_gb300.configs import ModelShape
    return ModelShape(f"wide-{hd}-{hq}-{hk}-{d}-{ff}", L, d, hq, hk, hd, ff, vocab, qk_norm=qk_norm, dtype="bf16",
                      rope_theta=500000.0)


def check(shape, n, max_rows=16):
    from paper_2602_20217_gb300 import synth
    from paper_2602_20217_gb300.model import Model
    prompt = synth.prompt_tokens(shape, n, seed=1)
    cfg, w = oracle_model(shape, seed=0)
    s = D.Session(cfg, w, n + 8)
    ref, _ = s.forward(prompt, 0)
    m = Model(shape, max_seq=n + 8, seed=0, max_rows=max_rows, hist_init_rows=min(8, max_rows))
    m.prefill(prompt)
    rows = min(n, max_rows)
    assert rel_err(m.logits(rows), ref[-rows:]) < 2e-2
    for layer in range(shape.n_layers):
        for which, full in (("k", s.k[layer]), ("v", s.v[layer])):
            got = m.kv(layer, 0, n, which)
            assert np.max(np.abs(got - full[:, :n])) <= 2e-2 * np.max(np.abs(full[:, :n])), (layer, which)
    first = m.logits(rows)
    m.prefill(prompt)                       # the same prompt again: bit for bit
    assert np.array_equal(first, m.logits(rows))
    m.close()


@pytest.mark.parametrize("n", [32, 33, 63, 127, 128, 129, 255, 256, 257, 400, 529, 784])
def test_tile_edges(n):
    check(shape_of(), n)


@pytest.mark.parametrize("hd,hq,hk,d,ff", [(64, 8, 2, 512, 1368), (64, 3, 3, 264, 72), (128, 16, 1, 520, 200),
                                           (128, 2, 2, 1032, 1032)])
def test_shapes(hd, hq, hk, d, ff):
    check(shape_of(hd=hd, qk_norm=hd == 64, hq=hq, hk=hk, d=d, ff=ff, vocab=333), 300)


def test_several_chunks():
    check(shape_of(L=2, hq=4, hk=2, ff=520), 2500)     # two even chunks of whole tiles, the second ragged


@pytest.mark.parametrize("max_rows", [2, 5])
def test_short_last_chunk(max_rows):
    check(shape_of(), 200, max_rows)
