"""Read-backs by several threads at once: right with more of them than the
process has staging areas, and side by side rather than one after the other
(four of 4.2 MB at once in 0.34 of the time they take in turn; behind one
another 0.86)."""
import threading
import time

import numpy as np
import pytest

from test_gpu_readout import _chain, _check

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _at_once(work, n):
    bad, gate = [], threading.Barrier(n + 1)

    def run(k):
        try:
            gate.wait()
            work(k)
        except BaseException as e:      # reported below, on the test's thread
            bad.append(e)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(n)]
    [t.start() for t in threads]
    gate.wait()
    t0 = time.perf_counter()
    [t.join() for t in threads]
    assert not bad, bad
    return time.perf_counter() - t0


def test_more_readers_than_staging_areas():
    chains = [_chain(20000 + 100 * k, 3000, 20, 3 + k, k) for k in range(12)]
    for _ in range(2):
        _at_once(lambda k: [_check(chains[k][0].posterior_mean(), chains[k][1], 3 + k) for _ in range(3)], 12)
    [ch.close() for ch, _ in chains]


def test_readers_do_not_queue():
    chains = [_chain(10000, 3000, 20, 5, k)[0] for k in range(4)]
    at_once = in_turn = np.inf
    for _ in range(8):
        at_once = min(at_once, _at_once(lambda k: [chains[k].posterior_mean() for _ in range(4)], 4))
        t0 = time.perf_counter()
        for ch in chains:
            for _ in range(4):
                ch.posterior_mean()
        in_turn = min(in_turn, time.perf_counter() - t0)
    assert at_once <= 0.65 * in_turn, (at_once, in_turn)
    [ch.close() for ch in chains]
