"""The selection kernels at the edges of their dispatch: knapsack
tables in shared memory and in the caller's scratch, capacities around whole
warps and odd item counts, cosine rows with and without 16-byte alignment.

Knapsack masks, weights and objectives are whole numbers and compared exactly;
cosines in fp32 carry d roundings of 2^-24 in each of three sums of the same
size: 1e-5 is above that for the widths here."""
import numpy as np
import pytest

from helpers import need_gpu
from oracle import select as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def solve(sims, units, budget):
    import torch

    from paper_2602_20217_gb300 import knapspec as ks
    n = len(sims)
    lat, _u = ks.latency(1, units=units)
    d = torch.as_tensor(np.asarray(sims, np.float32), device="cuda")
    mask = torch.zeros(n, dtype=torch.uint8, device="cuda")
    obj = torch.zeros(1, dtype=torch.float64, device="cuda")
    wts = torch.zeros(n, dtype=torch.int32, device="cuda")
    nb = ks.ks_select_scratch_bytes(n, budget)
    scratch = torch.empty(nb + 64, dtype=torch.uint8, device="cuda").fill_(0xA5)
    ks.ks_select_mask(lat, d, 100, n, budget, mask, obj, wts, scratch, nb, torch.cuda.current_stream())
    assert bool((scratch[nb:] == 0xA5).all())            # nothing past the scratch
    return mask.cpu().numpy(), float(obj.cpu()[0]), wts.cpu().numpy()


@pytest.mark.parametrize("n,budget,most", [(2, 0, 3), (2, 1, 3), (6, 31, 8), (6, 32, 8), (10, 63, 12), (64, 127, 4),
                                           (64, 128, 4), (128, 153, 2), (256, 255, 3), (30, 1023, 64), (30, 1024, 64),
                                           (128, 6000, 90), (256, 4000, 30), (256, 4800, 40), (40, 14000, 700),
                                           (12, 65535, 9000)])
def test_knapsack_capacities(n, budget, most):
    rng = np.random.default_rng(n * 100003 + budget)
    units = rng.integers(1, most + 1, n).astype(np.int32)
    sims = (1 - rng.integers(0, 40, n) / 64.0).astype(np.float32)      # many equal values: ties
    mask, obj, wts = solve(sims, units, budget)
    ref_mask, ref_total = S.knapsack(units, S.quantize_values(sims), budget)
    assert list(wts) == list(units)
    assert list(mask) == list(ref_mask)
    assert obj == ref_total / 2.0 ** 30


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("pairs,rows,d,extra,offset", [(1, 1, 1, 0, 0), (3, 4, 7, 0, 0), (2, 33, 64, 0, 0),
                                                       (5, 32, 128, 0, 1), (2, 31, 130, 2, 0), (4, 65, 512, 8, 0),
                                                       (2, 100, 4096, 4, 0), (2, 9, 4096, 0, 4),
                                                       (1, 64, 512, 0, 0), (3, 601, 131, 2, 1)])
def test_cosine_alignment(dtype, pairs, rows, d, extra, offset):
    import torch

    from paper_2602_20217_gb300 import knapspec as ks
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator().manual_seed(rows * 1009 + d)
    stride = rows * d + extra
    buf = torch.randn((pairs + 1) * stride + offset, generator=g).to(dt).cuda()
    x = buf[offset:]
    out = torch.zeros(pairs, device="cuda")
    ks.ks_cosine(x, x[stride:], ks.KS_DTYPE_F32 if dtype == "f32" else ks.KS_DTYPE_BF16, pairs, rows, d, stride, None,
                 out, torch.cuda.current_stream())
    ref = [float(torch.nn.functional.cosine_similarity(
        x[p * stride:p * stride + rows * d].double().view(rows, d),
        x[(p + 1) * stride:(p + 1) * stride + rows * d].double().view(rows, d), -1).mean()) for p in range(pairs)]
    assert np.max(np.abs(out.cpu().numpy() - ref)) < 1e-5
