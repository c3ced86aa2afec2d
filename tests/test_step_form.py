"""Which form a sparse part-step takes, read off the device bytes that
psgld_estimate_device_bytes counts for it (the form by units keeps the own
rows of both sides and its units' sums): on either side of the rule's lines,
at shapes that were measured in both forms.  CPU only."""
import pytest

from paper_1506_01418_gb300 import psgld as P


def _by_units(I, J, K, B, rho):
    """rho: entries of a part per row of either factor."""
    n, ldk = int(rho * B * (I + J) / 2), 4 * ((K + 3) // 4)
    light = 2 if I + J < 4864 else 8 if K <= 4 and min(I, J) < 9728 else 16
    held = 7 * (I + J) * ldk * 4 + 20 * 256 + 1216 * 8 + 64
    for rows in (I, J):
        held += (B * rows + 1) * 4 + 16 * (min(n // (light + 1), B * rows) + n // 512 + n // 128)
        held += (4 * ldk + 4) * (n // 512 + min(n // 128, rows))
    held += n * 20
    E = 32 if K <= 128 else 16 if K <= 256 else 8
    more = P.psgld_estimate_device_bytes(I, J, K, B, n) - held
    assert more in (0, 4 * n + 2 * 4 * 2 * (n // E + 1) * ldk)
    return more > 0


@pytest.mark.parametrize("I,J,K,B,rho,units", [
    (300000, 5000, 4, 16, 0.5, True), (300000, 5000, 4, 16, 2.0, False),       # 188 / 232; 267 / 211 us
    (480000, 18000, 8, 64, 0.5, True), (100000, 5000, 8, 8, 0.5, False),       # 1358 / 1703; 78 / 70
    (70000, 10000, 20, 32, 1.0, True), (30000, 5000, 20, 8, 1.0, False),       # 382 / 447; 73 / 66
    (70000, 10000, 36, 32, 4.0, True), (30000, 5000, 36, 8, 4.0, True),        # 828 / 910; 117 / 134
    (30000, 5000, 36, 8, 1.0, False),                                          # 105 / 93
    (75000, 75000, 100, 16, 2.0, False), (75000, 75000, 200, 16, 2.0, False),  # 1421 / 1195; 2605 / 2027
    (300000, 5000, 50, 16, 0.4, True), (70000, 10000, 50, 32, 7.8, False),
    (480000, 18000, 100, 64, 6.3, False)])
def test_form_at_measured_shapes(I, J, K, B, rho, units):
    assert _by_units(I, J, K, B, rho) == units
