"""Integrations of the request loop add FP32 pair terms in short runs.

Heavy particles in one point move together at (0, w, 0), massless ones start at rest at distance
1; eps^2 = 3. The heavy ones stay on their course and have the largest step, the massless ones
fall with M / 8: r^2 + eps^2 is 4 in FP32 throughout (the offset stays below 2^-12), every pair term
m / 8 and exact. The heavy masses are 1 or 1 + 2^-17 (times 2^-40), so an FP32 sum of up to 127
of them is exact and longer ones are not. The small steps' due sets are the massless particles;
with the sums exact their velocity is M t / 8 up to the jerk's part of the corrector, less than
dt^2 / 12 times the jerk's x component, 2^-29 of it. Only the first evaluation and the last
step, where all particles are due, come from other kernels (sums of 128 terms, 2^-26 of the
result and less after the share of one step). With a lane's whole share in one FP32 sum the 6000
particles were 2^-20 off."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,small", [(8192, 700), (6000, 900), (4097, 1300)])
def test_exact_sums_in_small_steps(nb, n, small):
    rng = np.random.default_rng(n)
    scale, w = 2.0 ** -40, 2.0 ** -8
    heavy = n - small
    m = np.zeros(n)
    m[small:] = scale * (1.0 + 2.0 ** -17 * rng.integers(0, 2, heavy))
    pos, vel = np.zeros((3, n)), np.zeros((3, n))
    pos[0, small:] = 1.0
    vel[1, small:] = w
    t = 2.0 ** -4
    with nb.Server(eta=2.0 ** -17, dt_max=t) as srv:
        r = srv.wait(srv.evolve(m, pos, vel, np.sqrt(3.0), t))
    assert r["block_steps"] > 4
    want = m.sum() / 8.0 * t
    assert np.abs(r["vel"][0, :small] / want - 1.0).max() < 2.0 ** -27
    np.testing.assert_array_equal(r["vel"][1, small:], np.full(heavy, w))
