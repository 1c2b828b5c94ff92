"""A workspace without the many-row passes' buffers is taken: prompts and the
hidden-state DP go through decode passes and agree with the oracle as they do
with the buffers (the comparisons and tolerances are those tests').  The sizes
are what the library asked for before it had those buffers."""
import pytest

import test_gpu_dp_states as states
import test_gpu_wide as wide
import test_gpu_wide_edges as edges
from helpers import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def take(monkeypatch, nbytes):
    from paper_2602_20217_gb300 import knapspec as ks
    asked = ks.ks_workspace_bytes

    def size(cfg):
        assert nbytes < asked(cfg)
        return nbytes
    monkeypatch.setattr(ks, "ks_workspace_bytes", size)


def test_prompt(monkeypatch):
    take(monkeypatch, 6591744)
    wide.check(wide.shape_of(), 300)


def test_states(monkeypatch):
    take(monkeypatch, 9410560)
    states.check(states.shape_of(128), 8, [5, 5], 64, states.UNITS8)


def test_tpt(monkeypatch):
    from paper_2602_20217_gb300.configs import ModelShape
    take(monkeypatch, 6270976)
    edges.check_tpt(ModelShape("narrow", 2, 512, 8, 2, 128, 1368, 333, dtype="bf16"), [5, 5], 8)


def test_too_little_is_refused(monkeypatch):
    from paper_2602_20217_gb300 import knapspec as ks
    from paper_2602_20217_gb300.model import Model
    take(monkeypatch, 1 << 20)          # less than the history and the RoPE table
    with pytest.raises(ks.KsError) as e:
        Model(wide.shape_of(), max_seq=308, seed=0)
    assert e.value.status == ks.KS_ERR_WORKSPACE
