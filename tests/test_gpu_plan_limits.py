"""Plan-table entries at the limits of a launch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_fp64_split_count_above_the_grid_limit(nb):
    """An FP64 tile entry's splits are units of 16 records: 65538 of them at N = 2^20 + 32, more
    than a grid has rows. An entry that asks for more is clamped, as one above the units is."""
    n = (1 << 20) + 32
    rng = np.random.default_rng(1)
    m, x, v = np.full(n, 1.0 / n), rng.standard_normal((n, 3)), rng.standard_normal((n, 3))
    with nb.System(m, x, v, variant="f64", eps=0.01) as sy:
        sy.predict(0.0)
        idx = np.array([17], dtype=np.int32)
        want = sy.force(idx)
        nb.nb_set_plan_table(sy.h, [(0, 1, 70000)])
        got = sy.force(idx)
        assert nb.nb_plan_for(sy.h, 1)[2] <= 65535
    for a, b in zip(got, want):
        # unit mass at unit distances: the magnitudes sum to about 1, and two orders of 2^20
        # terms differ by about 2^-53 x 2^10 = 1e-13 of that
        np.testing.assert_allclose(a, b, rtol=1e-11, atol=1e-11)
