"""How many FP32 terms the force kernels add before a sum goes into a double-single total.

Outside positions at the origin, every particle at (1, 0, 0), no softening: each pair adds the
particle's mass to the potential and to the x-acceleration, without rounding. The masses are 1
or 1 + 2^-18, so a sum of up to 63 of them is a 24-bit number and exact, and one of 64 and more
is not whenever it is odd. Sets of fewer than 4096 are exact if no FP32 sum, its two packed
halves together, is longer than the 32 terms of the scalar warp groups (kind 1)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _field(nb, n, ni, entry=None, grain=2.0 ** -18):
    rng = np.random.default_rng(n + ni)
    m = 1.0 + grain * rng.integers(0, 2, n)
    x = np.zeros((n, 3))
    x[:, 0] = 1.0
    with nb.System(m, x, np.zeros((n, 3)), variant="f32ds", eps=0.0, device=0) as sy:
        if entry:
            nb.nb_set_plan_table(sy.h, [entry] * 32)
        sy.predict(0.0)
        acc, jerk, pot = sy.force_ext(np.zeros((3, ni)), np.zeros((3, ni)))
    return m.sum(), acc, jerk, pot


@pytest.mark.parametrize("n", [2500, 20011, 65536])
@pytest.mark.parametrize("ni", [3, 17, 32, 33, 300, 1531, 2516, 4095])
@pytest.mark.parametrize("entry", [None, (1, 1, 2)])
def test_fp32_sums_of_due_sets_are_short(nb, n, ni, entry):
    total, acc, jerk, pot = _field(nb, n, ni, entry)
    np.testing.assert_array_equal(pot, np.full(ni, -total))
    np.testing.assert_array_equal(acc[0], np.full(ni, total))
    assert not acc[1:].any() and not jerk.any()


@pytest.mark.parametrize("n", [100, 200, 300, 400, 480])
@pytest.mark.parametrize("ni", [5, 33, 300, 480, 1531])
def test_fp32_sums_over_small_systems_are_shorter(nb, n, ni):
    """Up to 480 particles a lane of the warp groups adds 15 terms at most: with masses of 1 or
    1 + 2^-20 up to 15 are exact, and an odd sum of 16 and more is not."""
    total, acc, jerk, pot = _field(nb, n, ni, grain=2.0 ** -20)
    np.testing.assert_array_equal(pot, np.full(ni, -total))
    np.testing.assert_array_equal(acc[0], np.full(ni, total))
    assert not acc[1:].any() and not jerk.any()
