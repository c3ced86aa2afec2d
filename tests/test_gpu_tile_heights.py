"""The two-sided kernel whose items form their own mu keeps V in tiles as high
as the longest row piece (32, 64, 96 or 128 rows), and its epilogue warps skip
rows past the piece: the drift test of the dense path at the edges of each
height, pieces of two lengths (an odd number of rows in two pieces)."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import test_gpu_dense as dense


@pytest.mark.parametrize("rows", [31, 32, 33, 64, 65, 96, 97, 127, 128, 129])
@pytest.mark.parametrize("kernel", ["two_sided", "two_sided_bf16v"])
def test_drift_at_the_edges_of_the_tile_heights(monkeypatch, rows, kernel):
    monkeypatch.setitem(dense.DENSE, "edge", (2 * rows - 1, 150, 24, 2, 1.0, 1.0, 0, "poisson", 1e-3))
    dense.test_dense_part_step_drift_within_bf16_bound("edge", kernel)
