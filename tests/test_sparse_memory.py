"""Device memory of sparse contexts: psgld_estimate_device_bytes bounds what a
context holds however its entries fall into parts and whichever form its
part-step takes, and a load that finds no room beside the layout memory kept
from the load before gives that back and goes on."""
import numpy as np
import pytest

from paper_1506_01418_gb300 import psgld as P


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


# everything in one of 64 parts: a head and a tail slot of K floats for every
# 8 entries (K = 512) and side, beside the factors' seven FP32-sized copies
@pytest.mark.parametrize("I,J,K,B,nnz,E", [(1_000_000, 100_000, 512, 64, 34_500_000, 8),
                                           (600_000, 200_000, 388, 64, 46_000_000, 8),
                                           (300_000, 5000, 16, 16, 1_000_000, 32)])
def test_estimate_counts_a_part_with_every_entry(I, J, K, B, nnz, E):
    factors = 7 * (I + J) * K * 4
    slots = 2 * 2 * (nnz // E) * K * 4
    assert P.psgld_estimate_device_bytes(I, J, K, B, nnz) >= factors + slots


class Counter:
    """An allocator that counts live bytes and refuses to pass `limit`."""

    def __init__(self, torch):
        self.torch, self.live, self.limit, self.refused = torch, {}, None, 0

    def alloc(self, nbytes, stream):
        if self.limit is not None and self.held() + nbytes > self.limit:
            self.refused += 1
            return 0
        p = self.torch.cuda.caching_allocator_alloc(nbytes)
        self.live[p] = nbytes
        return p

    def free(self, ptr, stream):
        self.live.pop(ptr)
        self.torch.cuda.caching_allocator_delete(ptr)

    def held(self):
        return sum(self.live.values())


@pytest.fixture
def counter():
    c = Counter(_torch())
    P.psgld_set_allocator(c.alloc, c.free)
    yield c
    P.psgld_set_allocator(None)


def _cells(I, J, B, n, seed, diagonal):
    g = np.random.Generator(np.random.Philox(seed))
    if diagonal:   # within the B diagonal blocks: part 0
        r = g.integers(0, B, n)
        i0, i1, j0, j1 = r * I // B, (r + 1) * I // B, r * J // B, (r + 1) * J // B
        cell = (i0 + (g.random(n) * (i1 - i0)).astype(np.int64)) * J + j0 + (g.random(n) * (j1 - j0)).astype(np.int64)
    else:
        cell = g.integers(0, I * J, n)
    cell = np.unique(cell)
    return (cell // J).astype(np.int32), (cell % J).astype(np.int32), np.ones(len(cell), np.float32)


# by rows of many entries, of few; by units (few entries per row, wide rows)
@pytest.mark.gpu
@pytest.mark.parametrize("I,J,K,B,n", [(3000, 2000, 50, 8, 300000), (20000, 500, 8, 4, 50000),
                                       (150000, 3000, 16, 4, 400000), (6000, 3000, 512, 8, 100000)])
@pytest.mark.parametrize("diagonal", [False, True])
def test_estimate_bounds_what_a_sparse_context_holds(counter, I, J, K, B, n, diagonal):
    i, j, v = _cells(I, J, B, n, 1, diagonal)
    ch = P.PSGLD(I, J, K, B, 0.0, 1.0, prior_kind=P.PSGLD_PRIOR_GAUSSIAN)
    ch.set_data_coo(i, j, v)
    held, est = counter.held(), P.psgld_estimate_device_bytes(I, J, K, B, len(i))
    ch.close()
    assert not counter.live
    assert held <= est
    if diagonal:
        assert est <= 1.5 * held       # and is not far above it where one part has them all


@pytest.mark.gpu
def test_load_goes_on_without_the_kept_layout(counter):
    I, J, K, B = 4000, 3000, 4, 4
    many, few = _cells(I, J, B, 400000, 1, False), _cells(I, J, B, 220000, 2, False)

    def load(*sets, limit=None):
        ch = P.PSGLD(I, J, K, B, 0.0, 1.0, prior_kind=P.PSGLD_PRIOR_GAUSSIAN)
        for s in sets[:-1]:
            ch.set_data_coo(*s)
        counter.limit, counter.refused = limit, 0
        try:
            ch.set_data_coo(*sets[-1])
            return counter.held(), counter.refused
        finally:
            counter.limit = None
            ch.close()

    alone, _ = load(few)
    kept, _ = load(many, few)
    assert alone < kept                        # the larger layout's memory stayed
    # the entries' copies (12 bytes each) and the sort's scratch (24 and its
    # counts) fit beside this load's own layout, but not beside the kept one
    lo, hi = alone, 2 * kept + 100 * len(few[0])
    while hi - lo > 4096:                      # the least limit a load alone needs
        mid = (lo + hi) // 2
        try:
            load(few, limit=mid)
            hi = mid
        except P.PsgldError as e:
            assert e.status == P.PSGLD_ERR_OOM
            lo = mid
    held, refused = load(many, few, limit=hi)
    assert refused > 0 and held <= hi
