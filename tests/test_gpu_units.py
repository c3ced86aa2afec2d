"""The sparse part-step by units of entries, and the line between it and the
part-step by rows: large factors with few entries per row, few entries at
K > 96, and the contexts just past that line.

Held to the oracle by the suite's per-element tolerance of one FP32 step
(gpu_helpers.STEP_RTOL); sweeps on two streams, captured or not, and their
profiled one-stream form agree bit for bit."""
import numpy as np
import pytest

from gpu_helpers import Pair
from paper_1506_01418_gb300 import datagen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _entries(I, J, n, seed, crowded=0):
    """About n entries; the first `crowded` rows of column 0 and row 0 filled
    (rows that span many units), row 1 and column 1 empty."""
    g = np.random.Generator(np.random.Philox(seed))
    i, j = g.integers(0, I, n), g.integers(0, J, n)
    i = np.concatenate([i, np.arange(min(crowded, I)), np.zeros(min(crowded, J), np.int64)])
    j = np.concatenate([j, np.zeros(min(crowded, I), np.int64), np.arange(min(crowded, J))])
    keep = (i != 1) & (j != 1)
    cell = np.unique(i[keep] * J + j[keep])
    v = g.uniform(0.5, 5.0, len(cell)).astype(np.float32)
    return (cell // J).astype(np.int32), (cell % J).astype(np.int32), v


def _check(I, J, K, B, n, p=0.0, crowded=0, steps=None, **opts):
    i, j, v = _entries(I, J, n, seed=I + K, crowded=crowded)
    W0, H0 = datagen.init_factors(I, J, K, seed=K, scale=0.3, nonneg=p > 0)
    pr = Pair(I, J, K, B, p, 1.0, i, j, v, W0, H0, prior_kind=0 if p else 1, seed=5, eps=1e-5, **opts)
    for t in range(1, (steps or B) + 1):
        pr.step_and_check(t, W0, H0)
    pr.gpu.close()


# more than 2^19 float4 groups, below and past the entries per row of a part
# from which rows are taken (2 + 4 x padding, 1 + 4 x padding beyond K = 64)
@pytest.mark.parametrize("I,K,rho", [(190000, 9, 3.0), (190000, 9, 3.7), (140000, 16, 1.9), (140000, 16, 2.1),
                                     (110000, 17, 4.0), (70000, 32, 1.9), (60000, 33, 3.0), (60000, 47, 2.0),
                                     (45000, 64, 1.9), (45000, 64, 2.1), (30000, 96, 0.9), (30000, 96, 1.1)])
def test_large_factors_match_oracle(I, K, rho):
    J, B = 3000, 2
    _check(I, J, K, B, int(rho * B * (I + J) / 2), crowded=1000, steps=1)


# K > 96: below 384 K entries in a part (32 K beyond K = 256), and past it
@pytest.mark.parametrize("K,n", [(97, 1), (97, 7), (100, 600), (128, 20000), (129, 33), (256, 4000), (257, 2000),
                                 (512, 5000), (97, 60000), (129, 70000), (193, 110000), (257, 12000), (385, 16000),
                                 (512, 20000)])
def test_wide_factors_match_oracle(K, n):
    _check(700, 460, K, 1, n, crowded=300)


@pytest.mark.parametrize("p", [1.0, 1.5, 2.0])
def test_every_power_matches_oracle(p):
    _check(900, 640, 101, 3, 30000, p=p, crowded=400)


@pytest.mark.parametrize("opts", [dict(freeze_W=1), dict(freeze_H=1), dict(use_graphs=0)])
def test_options_match_oracle(opts):
    _check(600, 500, 101, 2, 20000, crowded=100, **opts)


@pytest.mark.parametrize("I,J,K", [(900, 640, 101), (180000, 60000, 100)])   # within L2, beyond it
def test_sweeps_agree_bit_for_bit(I, J, K):
    B = 3
    i, j, v = _entries(I, J, 40000, seed=1, crowded=500)
    W0, H0 = datagen.init_factors(I, J, K, seed=1, scale=0.3, nonneg=False)
    got = []
    for opts in (dict(use_graphs=1), dict(use_graphs=0), dict(profile=1)):
        pr = Pair(I, J, K, B, 0.0, 1.0, i, j, v, W0, H0, prior_kind=1, seed=5, eps=1e-5, **opts)
        pr.gpu.sweep(3)
        got.append(pr.gpu_factors())
        # data of the other form on the same context, then back
        k, m, x = _entries(I, J, 4000, seed=2)
        if I < 1000:
            k, m = np.divmod(np.arange(I * J), J)
            x = np.ones(I * J)
        for a, b, c in ((k, m, x), (i, j, v)):
            pr.gpu.set_data_coo(*(torch.as_tensor(z, dtype=d, device="cuda")
                                  for z, d in ((a, torch.int32), (b, torch.int32), (c, torch.float32))))
            pr.set_factors(W0, H0)
            pr.gpu.sweep(1)
        got.append(pr.gpu_factors())
        pr.gpu.close()
    for s in (0, 1):
        for W, H in got[2 + s::2]:
            assert np.array_equal(W, got[s][0]) and np.array_equal(H, got[s][1])
