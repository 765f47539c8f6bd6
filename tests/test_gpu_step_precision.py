"""Block steps of small systems add FP32 pair terms in short runs.

Heavy particles in one point move together at (0, w, 0), 20 massless ones start at rest at distance
1; eps^2 = 3. The heavy ones stay on their course and have the largest step, the massless ones fall
with M / 8: r^2 + eps^2 is 4 in FP32 throughout (the offset stays below 2^-12), every pair term m / 8
and exact. All heavy masses are 1 + 2^-18 (times 2^-40): an FP32 sum of up to 63 of them is exact,
and one of an odd number from 65 on (below 128) or from 129 on is not, by up to 2^-24. The sizes
give each of 16 parts of the system an odd number of 65 to 255 particles, so parts that are summed
in FP32 alone are off in the same direction. The small steps' due sets are the massless particles;
with the sums exact their velocity is M t / 8 up to the jerk's part of the corrector, less than
dt^2 / 12 times the jerk's x component, 2^-29 of it. Only the first evaluation and the last step, where
all particles are due, come from other kernels: 2^-24 at most, times the share of one step, 2^-5."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["f32", "f32ds"])
@pytest.mark.parametrize("n", [1040, 1296, 2500, 4080])
def test_exact_sums_in_small_steps(nb, n, variant):
    assert (n + 15) // 16 % 2 == 1
    small = 20
    scale, w = 2.0 ** -40, 2.0 ** -8
    m = np.zeros(n)
    m[small:] = scale * (1.0 + 2.0 ** -18)
    pos, vel = np.zeros((n, 3)), np.zeros((n, 3))
    pos[:small, 0] = 1.0
    vel[small:, 1] = w
    t = 2.0 ** -4
    with nb.System(m, pos, vel, variant=variant, eps=np.sqrt(3.0), eta=2.0 ** -23, dt_max=t) as sy:
        nb.nb_init(sy.h)
        st = sy.step(t)
        s = sy.state()
    assert st["block_steps"] >= 32 and st["fused_steps"] >= 31
    want = m.sum() / 8.0 * t
    assert np.abs(-s["vel"][0, :small] / want - 1.0).max() < 2.0 ** -27
    np.testing.assert_array_equal(s["vel"][1, small:], np.full(n - small, w))
