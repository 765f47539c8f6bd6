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


def _state_budget(nb, **cfg):
    """The least budget_bytes that nb_create accepts."""
    lo, hi = 1, 1 << 32
    while lo < hi:
        mid = (lo + hi) // 2
        try:
            nb.nb_destroy(nb.nb_create(nb.nb_config_default(device=0, budget_bytes=mid, **cfg)))
            hi = mid
        except nb.NBodyError as e:
            assert e.status == nb.NB_ERR_BUDGET
            lo = mid + 1
    return lo


@pytest.mark.parametrize("room", [1 << 17, 1 << 19, 1 << 21])
def test_forces_within_a_tight_budget(nb, room):
    """A budget with little room beside the state: the built-in plans split the j-range into as
    many parts as fit (1531 of 65536 would take 3.3 MB), and scratch that an earlier call
    took does not refuse a later one."""
    n = 65536
    rng = np.random.default_rng(2)
    m, x, v = np.full(n, 1.0 / n), rng.standard_normal((n, 3)), rng.standard_normal((n, 3))
    budget = _state_budget(nb, n_max=n, variant=nb.NB_F32DS) + room
    with nb.System(m, x, v, variant="f32ds", eps=0.01) as free, \
            nb.System(m, x, v, variant="f32ds", eps=0.01, budget_bytes=budget) as sy:
        free.predict(0.0)
        sy.predict(0.0)
        for ni in (3, 300, 1531, 40):
            idx = np.arange(0, 40 * ni, 40, dtype=np.int32)
            for a, b in zip(sy.force(idx), free.force(idx)):
                # FP32 pair terms in two orders of summation: a few FP32 roundings of the
                # largest result
                assert np.abs(a - b).max() <= 4e-6 * np.abs(b).max()
        sy.force_ext(x.T[:, :500].copy(), v.T[:, :500].copy())
