"""Log-likelihood and RMSE of sparse data against FP64 numpy: K around the
groups of four factor columns the kernel reads at a time, an odd K for the
FP64 sums' pairs, factors that are zero or subnormal (the integer widening
leaves them to the conversion instruction), and every form of the divergence.

Tolerance: both sides add the same FP64 terms in another order; K products
and nnz terms give a relative error of at most (K + nnz) 2^-53 of the sums of
magnitudes, held to 1e-11 of them here.
"""
import numpy as np
import pytest

from paper_1506_01418_gb300 import psgld as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 7, 16, 33, 50])
@pytest.mark.parametrize("p", [0.0, 1.0, 1.5, 2.0])
def test_sparse_log_lik_and_rmse_match_numpy(K, p):
    I, J, B, nnz = 211, 97, 3, 4000
    g = np.random.Generator(np.random.Philox(K * 10 + int(2 * p)))
    cell = np.sort(g.choice(I * J, size=nnz, replace=False))
    i, j = (cell // J).astype(np.int32), (cell % J).astype(np.int32)
    v = g.uniform(0.5, 5.0, nnz).astype(np.float32)
    W = g.uniform(0.1, 1.5, (I, K)).astype(np.float32)
    H = g.uniform(0.1, 1.5, (J, K)).astype(np.float32)
    W[::7, 0] = 0.0
    W[1::7, K - 1] = np.float32(1e-41)          # subnormal
    H[::5, K - 1] = np.float32(3e-40)
    ch = P.PSGLD(I, J, K, B, p, 0.7, seed=1, eps=1e-4, mu_min=1e-2)
    ch.set_data_coo(i, j, v)
    ch.set_factors(W, H)
    n = 3
    sW, sH = g.uniform(0.3, 3.0, (I, K)), g.uniform(0.3, 3.0, (J, K))
    ch.set_state((sW, sW * sW, sH, sH * sH, np.array([n * B, n, n], np.int64)))

    v64 = v.astype(np.float64)
    mu = np.einsum("nk,nk->n", W.astype(np.float64)[i], H.astype(np.float64)[j])
    m, b = (np.maximum(mu, 1e-2) if p > 0 else mu), 2.0 - p
    if b == 2.0:
        terms = [0.5 * (v64 - m) ** 2]
    elif b == 1.0:
        terms = [v64 * np.log(v64 / m), -v64, m]
    elif b == 0.0:
        terms = [v64 / m, -np.log(v64 / m), -np.ones(nnz)]
    else:
        terms = [v64 ** b / (b * (b - 1)), -v64 * m ** (b - 1) / (b - 1), m ** b / b]
    size = sum(np.abs(t) for t in terms).sum() / 0.7
    assert abs(ch.log_lik() + sum(terms).sum() / 0.7) <= 1e-11 * size

    for use_mean, mean in ((False, mu), (True, np.einsum("nk,nk->n", sW[i] / n, sH[j] / n))):
        want = np.sqrt(np.mean((v64 - mean) ** 2))
        scale = np.sqrt(np.mean((np.abs(v64) + np.abs(mean)) ** 2))
        assert abs(ch.rmse(use_mean) - want) <= 1e-11 * scale
    ch.close()
