"""The sparse part-step's shares of a row: a team, a warp or a block's chunks,
by the row's entries in the part, at the edges of each range, for every lane
layout of a factor row (K around the group counts where it changes).

One part holds everything (B = 1); rows have 0, 1, 2, 3, 15, 16, 17, 127, 128,
129, 511, 512, 513 and 1025 entries, column 0 has one in every row (several
chunks).  4000 rows give the rows of at most 16 entries to teams, 1100 rows
those of at most 2.  Held to the oracle by the suite's per-element tolerance
of one FP32 step (gpu_helpers.STEP_RTOL), twice from the same factors, which
must agree bit for bit (chunks are added in order, whichever arrives last)."""
import numpy as np
import pytest

from gpu_helpers import Pair
from paper_1506_01418_gb300 import datagen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

DEGREES = [0, 1, 2, 3, 15, 16, 17, 127, 128, 129, 511, 512, 513, 1025]


def _entries(I, J, seed):
    g = np.random.Generator(np.random.Philox(seed))
    i, j = [], []
    for row in range(I):
        # the listed degrees at both ends of the rows, column 0 alone between
        at = row if row < len(DEGREES) else row - (I - len(DEGREES))
        n = DEGREES[at] if 0 <= at < len(DEGREES) else 1
        cols = np.concatenate([[0], 1 + g.choice(J - 1, size=max(n - 1, 0), replace=False)])[:n]
        i += [row] * n
        j += sorted(cols)
    v = g.uniform(0.5, 5.0, len(i))
    return np.array(i, np.int32), np.array(j, np.int32), v.astype(np.float32)


@pytest.mark.parametrize("K", [1, 4, 5, 8, 9, 16, 17, 32, 33, 50, 64, 65, 100, 128, 129, 192, 193, 256, 257, 384, 385,
                               512])
@pytest.mark.parametrize("I", [1100, 4000])
def test_rows_of_every_length_match_oracle(I, K):
    J = 1100
    i, j, v = _entries(I, J, seed=I + K)
    W0, H0 = datagen.init_factors(I, J, K, seed=K, scale=0.3, nonneg=False)
    pr = Pair(I, J, K, 1, 0.0, 1.0, i, j, v, W0, H0, prior_kind=1, seed=5, eps=1e-5)
    W1, H1 = pr.step_and_check(1)
    pr.set_factors(W0, H0)
    pr.gpu.part_step(1)
    W2, H2 = pr.gpu_factors()
    assert np.array_equal(W1, W2) and np.array_equal(H1, H2)
    pr.gpu.close()


@pytest.mark.parametrize("p", [1.0, 1.5, 2.0])
def test_rows_without_entries_ignore_the_rest_of_their_warp(p):
    """A row without entries moves by prior and noise alone, whatever its
    neighbours' entries are (here: mu below mu_min, so large factors e)."""
    I, J, K, B = 6000, 300, 13, 3
    g = np.random.Generator(np.random.Philox(9))
    cell = np.unique(g.integers(0, (I // 2) * J, 30000))
    i, j = (2 * (cell // J)).astype(np.int32), (cell % J).astype(np.int32)   # odd rows: none
    v = g.uniform(0.5, 5.0, len(i)).astype(np.float32)
    W0, H0 = datagen.init_factors(I, J, K, seed=1, scale=1e-3, nonneg=True)
    pr = Pair(I, J, K, B, p, 1.0, i, j, v, W0, H0, prior_kind=0, seed=5, eps=1e-9)
    for t in range(1, B + 1):
        pr.step_and_check(t, W0, H0)
    pr.gpu.close()
