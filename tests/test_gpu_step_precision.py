"""Block steps of small systems add FP32 pair terms in short runs.

Heavy particles in one point move together at (0, w, 0), 20 massless ones start at rest at distance
1; eps^2 = 3. The heavy ones stay on their course and have the largest step; the massless ones are
pulled by M / 8, so weakly that their steps are below half an ulp of x and it stays 1 in FP64 (FP32
cuts positions off, and 1 less one ulp would be 2^-24 less). r^2 + eps^2 is 4 in FP32 throughout (the
offset stays below 2^-12), every pair term m / 8 and exact. All heavy masses are 1 + 2^-18 (times
2^-60): an FP32 sum of up to 63 of them is exact, and one of an odd number from 65 on (below 128) or
from 129 on is not, by up to 2^-24. The sizes give each of 16 parts of the system an odd number of 65
to 123 particles, so parts that are summed in FP32 alone are off in the same direction. The small
steps' due sets are the massless particles. At half of dt_max, where the heavy ones are not due, their
acceleration is the sum of a small step: with the terms' sums exact it is M / 8. (Not their velocity:
the first evaluation of all particles is another kernel's, which for f32 adds in plain FP32 and may
lose the 2^-18 of every mass.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["f32", "f32ds"])
@pytest.mark.parametrize("n", [1040, 1296, 1904, 1968])
def test_exact_sums_in_small_steps(nb, n, variant):
    assert (n + 15) // 16 % 2 == 1
    small = 20
    scale, w = 2.0 ** -60, 2.0 ** -8
    m = np.zeros(n)
    m[small:] = scale * (1.0 + 2.0 ** -18)
    pos, vel = np.zeros((n, 3)), np.zeros((n, 3))
    pos[:small, 0] = 1.0
    vel[small:, 1] = w
    t = 2.0 ** -4
    with nb.System(m, pos, vel, variant=variant, eps=np.sqrt(3.0), eta=2.0 ** -17, dt_max=t) as sy:
        nb.nb_init(sy.h)
        st = sy.step(t / 2)
        s = sy.state()
    assert st["block_steps"] >= 4 and st["fused_steps"] == st["block_steps"]
    assert (s["t"][:small] == t / 2).all() and (s["t"][small:] == 0.0).all()
    np.testing.assert_array_equal(s["pos"][0, :small], np.ones(small))
    want = m.sum() / 8.0
    assert np.abs(-s["acc"][0, :small] / want - 1.0).max() < 2.0 ** -27
    np.testing.assert_array_equal(s["vel"][1, small:], np.full(n - small, w))
