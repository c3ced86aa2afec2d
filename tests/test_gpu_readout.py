"""Posterior means and variances from given sums: below and above the sizes
that go through the staging area, rows that do not fill its halves, K off the
multiple of four, arrays left out, no samples, and several contexts read by
several threads at once.  The host forms the same divisions in FP64; the
variance may differ by the rounding of one product (fused or not): 2^-52 of
mean^2."""
import threading

import numpy as np
import pytest

from paper_1506_01418_gb300 import psgld as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _chain(I, J, K, n, seed):
    g = np.random.Generator(np.random.Philox(seed))
    ch = P.PSGLD(I, J, K, 2, 0.0, 1.0, prior_kind=P.PSGLD_PRIOR_GAUSSIAN)
    ch.set_data_coo(np.arange(2, dtype=np.int32), np.arange(2, dtype=np.int32), np.ones(2, np.float32))
    ch.set_factors(np.zeros((I, K), np.float32), np.zeros((J, K), np.float32))
    sums = []
    for rows in (I, J):
        m = g.standard_normal((rows, K))
        sums += [m * n, (m * m + g.random((rows, K))) * n]
    ch.set_state((*sums, np.array([2 * n, n, n], np.int64)))
    return ch, sums


def _check(got, sums, n):
    assert got[4] == n
    for k, (s, s2) in enumerate(((sums[0], sums[1]), (sums[2], sums[3]))):
        m = s / n
        assert np.array_equal(got[2 * k], m)
        assert np.all(np.abs(got[2 * k + 1] - (s2 / n - m * m)) <= 2.0 ** -52 * (m * m + s2 / n))


@pytest.mark.parametrize("I,J,K", [(5, 4, 1), (300, 200, 13), (2048, 32, 16), (30011, 517, 33), (9000, 40000, 50),
                                   (3, 2000, 512), (600000, 2, 3)])
def test_moments_match_numpy(I, J, K):
    ch, sums = _chain(I, J, K, 7, I)
    _check(ch.posterior_mean(), sums, 7)
    Wv = np.full((I, K), np.nan)
    assert P.psgld_posterior_mean(ch.ctx, None, Wv, None, None) == 7          # one array alone
    assert np.array_equal(Wv, ch.posterior_mean()[1])
    ch.set_data_coo(np.arange(2, dtype=np.int32), np.arange(2, dtype=np.int32), np.ones(2, np.float32))
    assert all(not np.any(x) for x in ch.posterior_mean()[:4])                # no samples: zeros
    ch.close()


def test_contexts_read_by_threads_at_once():
    chains = [_chain(20000 + 1000 * k, 3000, 40, 3 + k, k) for k in range(4)]
    bad = []

    def read(k):
        try:
            for _ in range(3):
                _check(chains[k][0].posterior_mean(), chains[k][1], 3 + k)
        except BaseException as e:      # reported below, on the test's thread
            bad.append(e)

    threads = [threading.Thread(target=read, args=(k,)) for k in range(4)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not bad, bad
    [ch.close() for ch, _ in chains]
