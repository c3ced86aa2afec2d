"""dense_path = 1: the two-sided kernel (the chain of dense_path = 2, bit for
bit), and, for blocks the single-pass kernel takes, that one when V's tiles
find no memory (the chain of dense_path = 3)."""
import numpy as np
import pytest

from paper_1506_01418_gb300 import datagen
from paper_1506_01418_gb300 import psgld as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _chain(path, I, J, K, B, **opts):
    V, _, _ = datagen.dense_gamma(I, J, 4, seed=3)
    W0, H0 = datagen.init_factors(I, J, K, seed=4, scale=0.5)
    c = P.PSGLD(I, J, K, B, 1.0, 1.0, seed=9, eps=1e-5, dense_path=path, **opts)
    c.set_data_dense(torch.from_numpy(V).cuda())
    c.set_factors(torch.from_numpy(W0).cuda(), torch.from_numpy(H0.T.copy()).cuda())
    c.sweep(2)
    out = [x.cpu().numpy() for x in c.get_factors()]
    c.close()
    return out


@pytest.mark.parametrize("I,J,K,B", [(100, 90, 8, 1), (257, 600, 16, 8), (129, 300, 100, 1), (640, 333, 128, 5)])
def test_auto_is_the_two_sided_chain(I, J, K, B):
    for a, b in zip(_chain(1, I, J, K, B), _chain(2, I, J, K, B)):
        assert np.array_equal(a, b)


def test_auto_without_memory_for_the_tiles_is_the_single_pass_chain():
    I, J, K, B = 257, 600, 16, 3                    # blocks of at most 128 rows
    want = _chain(3, I, J, K, B)
    live, refused = {}, []

    def alloc(nbytes, stream):
        if nbytes > 4 * I * J:                      # V itself fits, its padded tiles do not
            refused.append(nbytes)
            return 0
        t = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
        at = (t.data_ptr() + 255) & ~255
        live[at] = t
        return at

    P.psgld_set_allocator(alloc, lambda ptr, stream: live.pop(ptr))
    try:
        got = _chain(1, I, J, K, B)
    finally:
        P.psgld_set_allocator(None)
    assert refused and not live
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
