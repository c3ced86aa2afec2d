"""Sparse part-steps where one of several parts holds nearly every entry
(block-diagonal data: clustered users and items), in every form the sparse
part-step takes: rows of many and of few entries, wide rows.
The other parts are empty or hold a single entry.  Held to the oracle by the
suite's per-element tolerance of one FP32 step (gpu_helpers.STEP_RTOL)."""
import numpy as np
import pytest

from gpu_helpers import Pair
from paper_1506_01418_gb300 import datagen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _diagonal(I, J, B, n, seed):
    """n entries drawn in the diagonal blocks (part 0), one in part 1."""
    g = np.random.Generator(np.random.Philox(seed))
    r = g.integers(0, B, n)
    i0, i1 = r * I // B, (r + 1) * I // B
    j0, j1 = r * J // B, (r + 1) * J // B
    cell = (i0 + (g.random(n) * (i1 - i0)).astype(np.int64)) * J + j0 + (g.random(n) * (j1 - j0)).astype(np.int64)
    cell = np.unique(np.append(cell, J // B))          # row 0, first column of piece 1
    v = g.uniform(0.5, 5.0, len(cell)).astype(np.float32)
    return (cell // J).astype(np.int32), (cell % J).astype(np.int32), v


# 300 x 200: rows of many entries; 150000 rows: few entries per row, by units;
# K = 512: by units for its few entries in an average part
@pytest.mark.parametrize("I,J,K,B,n", [(300, 200, 50, 4, 9000), (150000, 3000, 16, 3, 250000),
                                       (2000, 900, 512, 6, 12000), (2000, 900, 128, 6, 30000)])
def test_all_entries_in_one_part(I, J, K, B, n):
    i, j, v = _diagonal(I, J, B, n, seed=I + K)
    W0, H0 = datagen.init_factors(I, J, K, seed=K, scale=0.3, nonneg=False)
    pr = Pair(I, J, K, B, 0.0, 1.0, i, j, v, W0, H0, prior_kind=1, seed=5, eps=1e-5)
    for t in range(1, B + 1):
        pr.step_and_check(t, W0, H0)
    pr.gpu.close()
