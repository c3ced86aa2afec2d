"""The entry layout from entries in any order: row-major input (the parts'
digits alone are sorted), shuffled input (columns, then rows of parts) and
row-major input with its last two entries exchanged give the same layouts,
which are numpy's, and the same chain; more than 256 parts take two digits.
Host and device arrays, reloads into the same context (smaller and larger,
its memory kept), duplicates and bad indices in either order."""
import numpy as np
import pytest

from paper_1506_01418_gb300 import datagen
from paper_1506_01418_gb300 import psgld as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _entries(I, J, nnz, seed):
    g = np.random.Generator(np.random.Philox(seed))
    cell = np.sort(g.choice(I * J, size=nnz, replace=False))
    return (cell // J).astype(np.int32), (cell % J).astype(np.int32), g.uniform(1, 5, nnz).astype(np.float32), g


def _check(ch, I, J, B, i, j):
    piece = lambda x, n: ((x.astype(np.int64) + 1) * B - 1) // n
    part = (piece(j, J) - piece(i, I)) % B
    for s in range(B):
        m = part == s
        order = np.lexsort((j[m], i[m]))
        ptr, cols = P.psgld_part_layout(ch.ctx, s, I)
        assert np.array_equal(cols, j[m][order]), s
        assert np.array_equal(ptr, np.concatenate([[0], np.cumsum(np.bincount(i[m], minlength=I))])), s


@pytest.mark.parametrize("I,J,B,nnz", [(50, 40, 1, 300), (700, 300, 7, 20000), (900, 700, 300, 50000),
                                       (5000, 3000, 16, 4096 * 9 + 1), (9, 8, 8, 72), (300, 200, 5, 1)])
def test_layout_of_ordered_and_shuffled_entries(I, J, B, nnz):
    i, j, v, g = _entries(I, J, nnz, I + B)
    mix = g.permutation(nnz)
    swap = np.arange(nnz)
    if nnz > 1:
        swap[[-1, -2]] = swap[[-2, -1]]
    W0, H0 = datagen.init_factors(I, J, 6, seed=2, scale=0.4)
    out = []
    for order, host in ((np.arange(nnz), False), (mix, False), (swap, True)):
        a = [np.ascontiguousarray(x[order]) for x in (i, j, v)]
        if not host:
            a = [torch.from_numpy(x).cuda() for x in a]
        ch = P.PSGLD(I, J, 6, B, 1.0, 1.0, seed=3, eps=1e-5)
        ch.set_data_coo(*a)
        _check(ch, I, J, B, i, j)
        ch.set_factors(W0, np.ascontiguousarray(H0.T))
        ch.sweep(2)
        out.append([x.cpu().numpy() for x in ch.get_factors()])
        ch.close()
    for o in out[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(o, out[0]))


def test_reloads_into_one_context():
    I, J, B = 600, 400, 4
    ch = P.PSGLD(I, J, 5, B, 0.0, 1.0, prior_kind=P.PSGLD_PRIOR_GAUSSIAN, seed=3, eps=1e-5)
    for nnz in (20000, 19000, 500, 60000, 59999):
        i, j, v, _ = _entries(I, J, nnz, nnz)
        ch.set_data_coo(i, j, v)
        _check(ch, I, J, B, i, j)
    ch.close()


@pytest.mark.parametrize("shuffled", [False, True])
def test_bad_entries_are_refused_and_the_context_takes_others(shuffled):
    I, J = 100, 80
    i, j, v, g = _entries(I, J, 2000, 1)
    order = g.permutation(2001) if shuffled else np.argsort(np.append(i, i[700]) * J + np.append(j, j[700]), kind="stable")
    dup = [np.ascontiguousarray(np.append(x, x[700])[order]) for x in (i, j, v)]
    ch = P.PSGLD(I, J, 4, 2, 1.0, 1.0)
    for bad, what in ((dup, "duplicate"), ([np.where(np.arange(2000) == 1999, I, i).astype(np.int32), j, v], "range"),
                      ([i, np.where(np.arange(2000) == 0, -1, j).astype(np.int32), v], "range"),
                      ([i, j, np.where(np.arange(2000) == 5, np.nan, v).astype(np.float32)], "finite")):
        with pytest.raises(P.PsgldError) as e:
            ch.set_data_coo(*bad)
        assert e.value.status == P.PSGLD_ERR_ARG and what in str(e.value)
    ch.set_data_coo(i, j, v)
    _check(ch, I, J, 2, i, j)
    ch.close()
