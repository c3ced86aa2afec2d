"""Read-backs on either side of the size from which moments go through the
staging area (1.5 MB), into used and into new memory: right, and not slower
into new memory than getting its pages explains (0.9 MB: 1.5 times; device
copies straight into new pages took 6 times)."""
import mmap
import time

import numpy as np
import pytest

from paper_1506_01418_gb300 import psgld as P
from test_gpu_readout import _chain, _check

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("rows", [98303, 98304, 98305, 60000, 20])   # of one FP64 moment of each factor, K = 1
def test_moments_around_the_staging_size(rows):
    # mean and variance of rows / 2 values a factor: 16 bytes a row
    I = rows // 2
    ch, sums = _chain(I, rows - I, 1, 7, rows)
    _check(ch.posterior_mean(), sums, 7)
    ch.close()


def test_new_memory_costs_its_pages_and_no_more():
    I, J, K = 2600, 900, 16                                          # 0.9 MB
    ch, _ = _chain(I, J, K, 7, 1)

    def new(n):
        return np.frombuffer(mmap.mmap(-1, 8 * n * K), dtype=np.float64).reshape(n, K)

    def t(arrays):
        t0 = time.perf_counter()
        P.psgld_posterior_mean(ch.ctx, *arrays)
        return time.perf_counter() - t0

    used = [np.ones((n, K)) for n in (I, I, J, J)]
    again = min(t(used) for _ in range(20))
    fresh = min(t([new(n) for n in (I, I, J, J)]) for _ in range(20))
    assert fresh <= 3 * again, (fresh, again)
    ch.close()
