"""The sparse part-step by units of entries with BF16-gathered factors: large
factors with few entries per row, for lane layouts of one group, of two and
of padded rows, and a context by rows beside them.  Each step's drift is held
to the first-order BF16 bound of test_gpu_sparse_bf16; the second step reads
the copies that the first one's update wrote.  Captured, direct and profiled
(one-stream) sweeps agree bit for bit."""
import numpy as np
import pytest

import oracle
from gpu_helpers import Pair, recovered_drift
from paper_1506_01418_gb300 import datagen
from test_gpu_sparse_bf16 import _sparse_bound

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

EPS, SEED, B = 1e-3, 7, 2


def _pair(I, J, K, rho, **opts):
    g = np.random.Generator(np.random.Philox(I + K))
    n = int(rho * B * (I + J) / 2)
    cell = np.unique(np.concatenate([g.integers(0, I * J, n), np.arange(0, 900 * J, J)]))   # column 0: a row of many units
    i, j = (cell // J).astype(np.int32), (cell % J).astype(np.int32)
    v = g.uniform(0.5, 5.0, len(cell)).astype(np.float32)
    W0, H0 = datagen.init_factors(I, J, K, seed=K, scale=0.3, nonneg=False)
    return Pair(I, J, K, B, 0.0, 1.0, i, j, v, W0, H0, prior_kind=1, seed=SEED, eps=EPS, gather_bf16=1, **opts)


@pytest.mark.parametrize("I,J,K,rho", [(264000, 2000, 4, 0.4), (264000, 2000, 7, 0.3), (264000, 2000, 12, 0.5),
                                       (264000, 2000, 33, 0.4), (264000, 2000, 72, 0.4), (70000, 2000, 20, 1.0),
                                       (70000, 2000, 23, 1.5), (70000, 2000, 33, 0.5)])
def test_drift_within_the_bf16_bound(I, J, K, rho):
    pr = _pair(I, J, K, rho)
    for t in (1, 2):
        W0, H0 = pr.orc.get_factors()
        D_W, D_H = pr.orc.drift(t)
        bW, bH = _sparse_bound(pr.i, pr.j, pr.v.astype(np.float32), W0, H0, t, B, 0.0, 1.0, pr.orc.scale(t))
        pr.gpu.part_step(t)
        Wg, Hg = pr.gpu_factors()
        zW = oracle.noise_matrix(SEED, t, 0, I, K)
        zH = oracle.noise_matrix(SEED, t, 1, J, K).T
        for xg, x0, z, D, bnd, what in ((Wg, W0, zW, D_W, bW, "W"), (Hg, H0, zH, D_H, bH, "H")):
            Dg, mask, rec = recovered_drift(xg.astype(np.float64), x0, z, D, EPS, False)
            err = np.abs(Dg - D)
            assert not (mask & (err > bnd + rec)).any(), (t, what, float((err - bnd - rec).max()))
            active = mask & (bnd > 0)
            assert np.sqrt(np.mean(D[active] ** 2)) > 4 * np.sqrt(np.mean(bnd[active] ** 2)), (t, what)
        pr.sync_oracle_to_gpu()
    pr.gpu.close()


def test_sweeps_agree_bit_for_bit():
    got = []
    for opts in (dict(use_graphs=1), dict(use_graphs=0), dict(profile=1)):
        pr = _pair(264000, 2000, 12, 0.4, **opts)
        pr.gpu.sweep(3)
        got.append(pr.gpu_factors())
        pr.gpu.close()
    for W, H in got[1:]:
        assert np.array_equal(W, got[0][0]) and np.array_equal(H, got[0][1])


def test_a_frozen_factor_stays_and_the_other_moves_as_without():
    pr, free = _pair(70000, 2000, 20, 1.0, freeze_H=1), _pair(70000, 2000, 20, 1.0)
    H0 = pr.gpu_factors()[1]
    pr.gpu.part_step(1)
    free.gpu.part_step(1)
    W, H = pr.gpu_factors()
    assert np.array_equal(H, H0) and np.array_equal(W, free.gpu_factors()[0])
    pr.gpu.close()
    free.gpu.close()
