"""Sizes of the device workspace (no GPU): small models take little, and the
partial sums of tiles cut along K (38 MiB) are taken only by models whose
projections can have such tiles, those with more than 7680 inputs."""
import os
import shutil

import pytest

MIB = 1 << 20


@pytest.fixture(scope="module")
def size():
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    from paper_2602_20217_gb300 import build, knapspec as ks
    from paper_2602_20217_gb300.configs import ModelShape
    build.build()

    def size(L, d, hq, hk, hd, ff, vocab, max_seq):
        return ks.ks_workspace_bytes(ks.make_config(ModelShape("w", L, d, hq, hk, hd, ff, vocab), max_seq))
    return size


def test_small_models_take_little(size):
    assert size(1, 64, 1, 1, 64, 128, 100, 64) < 3.9 * MIB
    assert size(2, 512, 8, 2, 128, 1368, 2000, 256) < 8 * MIB


@pytest.mark.parametrize("kw", [dict(ff=7680), dict(hq=60, hk=4), dict(d=7680)])
def test_partials_only_where_tiles_can_be_cut(size, kw):
    base = dict(L=1, d=512, hq=4, hk=4, hd=128, ff=512, vocab=1000, max_seq=256)
    a = size(**{**base, **kw})
    more = {"ff": dict(ff=7688), "hq": dict(hq=64, hk=4), "d": dict(d=7688)}[next(iter(kw))]
    b = size(**{**base, **kw, **more})
    assert a < 60 * MIB and b - a > 30 * MIB
