"""Entry arrays in device memory at any byte address: aligned ones are read in
place, the others through a copy; the same layout, hence the same part-step,
bit for bit."""
import ctypes as C

import numpy as np
import pytest

from paper_1506_01418_gb300 import datagen
from paper_1506_01418_gb300 import psgld as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _at(x, offset):
    """x's bytes in device memory, `offset` bytes past an allocation's start."""
    b = x.tobytes()
    buf = torch.zeros(len(b) + 16, dtype=torch.uint8, device="cuda")
    buf[offset:offset + len(b)] = torch.frombuffer(bytearray(b), dtype=torch.uint8).cuda()
    return buf, buf.data_ptr() + offset


def test_entries_at_any_address():
    I, J, K, B, n = 70, 50, 6, 3, 400
    g = np.random.Generator(np.random.Philox(1))
    cell = g.permutation(I * J)[:n]                      # not in row-major order
    arrays = (cell // J).astype(np.int32), (cell % J).astype(np.int32), g.uniform(1, 5, n).astype(np.float32)
    W0, H0 = datagen.init_factors(I, J, K, seed=1, scale=0.3, nonneg=False)
    got = []
    for offsets in ((0, 0, 0), (4, 8, 12), (1, 0, 0), (0, 2, 0), (0, 0, 3), (3, 1, 2)):
        ch = P.PSGLD(I, J, K, B, 0.0, 1.0, prior_kind=P.PSGLD_PRIOR_GAUSSIAN, seed=5, eps=1e-4)
        held = [_at(x, o) for x, o in zip(arrays, offsets)]
        torch.cuda.synchronize()
        s = P.load().psgld_set_data_coo(ch.ctx, C.c_int64(n), *(C.c_void_p(p) for _, p in held), None)
        assert s == P.PSGLD_OK
        ch.set_factors(torch.from_numpy(W0).cuda(), torch.from_numpy(H0.T.copy()).cuda())
        ch.part_step(1)
        W, Ht = ch.get_factors()
        torch.cuda.synchronize()
        got.append((W.cpu().numpy(), Ht.cpu().numpy()))
        ch.close()
    for W, Ht in got[1:]:
        assert np.array_equal(W, got[0][0]) and np.array_equal(Ht, got[0][1])
