"""Bytes that the bench counts for a launch of a Kaczmarz level in FP32 tiles."""
import pytest

import bench


@pytest.mark.parametrize("launches,separate", [(1, False), (2, False), (4, False), (2, True), (4, True)])
def test_kaczmarz_bytes_follow_the_launches_of_a_pass(launches, separate):
    """The sum over a V-cycle's launches, written out: u (8 bytes complex) in except from the zero guess and out, f,
    k h (4), and with the transfers in the same launches the coarse f and e, a quarter of a level each."""
    level, iterations = 2, 2
    per = {("kacz_sweep", level): [0.05] * (4 * launches * iterations)}
    if separate:
        per[("restrict_residual", level)] = [0.01] * (2 * iterations)
        per[("prolong_add", level)] = [0.01] * (2 * iterations)
    down = sum((0 if q == 0 else 8) + 8 + 4 + 8 for q in range(launches)) + (0 if separate else 8 / 4)
    up = launches * (8 + 8 + 4 + 8) + (0 if separate else 8 / 4)
    want = (down + up) / (2 * launches)
    assert bench.launch_bytes_per_node(per, "kacz_sweep", level, True) == pytest.approx(want)
    rates = bench.sweep_rates(per, True, 6669.2, 4096)
    assert rates["kacz_sweep@L2"]["gbs"] == pytest.approx(want * 1025**2 / 0.05e-3 / 1e9, abs=0.1)
