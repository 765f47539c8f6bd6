"""The request loop around its integrations' cluster launches: failures, counters, requests beside
them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _overflowing(n=50):
    """Finite at the start; one particle is so fast that its distances overflow FP32 after the
    first, smallest step (2^-30): the pair terms of that step are not finite."""
    rng = np.random.default_rng(4)
    m, pos, vel = np.full(n, 1.0 / n), rng.standard_normal((3, n)), np.zeros((3, n))
    vel[0, 7] = 1e30
    return m, pos, vel


def test_an_error_ends_the_integration_at_its_step(nb):
    with nb.Server(dt_max=1.0 / 16) as srv:
        r = srv.wait(srv.evolve(*_overflowing(), 0.01, 1.0))
        assert r["status"] == nb.NB_STATUS_ERROR and r["error"] == nb.NB_ERR_NONFINITE
        assert r["block_steps"] <= 1
        # the loop goes on
        rng = np.random.default_rng(5)
        ok = srv.wait(srv.evolve(np.full(64, 1 / 64.0), rng.standard_normal((3, 64)),
                                 np.zeros((3, 64)), 0.1, 1.0 / 16))
        assert ok["status"] == nb.NB_STATUS_DONE


def test_busy_time_counts_cluster_launches(nb):
    """One integration of 500 particles: nearly all of its time is its cluster launches'."""
    rng = np.random.default_rng(6)
    m, pos, vel = np.full(500, 1 / 500.0), rng.standard_normal((3, 500)), np.zeros((3, 500))
    with nb.Server(dt_max=1.0 / 16) as srv:
        srv.wait(srv.evolve(m, pos, vel, 0.03, 1.0 / 16))  # the handle and the kernels are there
        before = srv.stats()["busy_s"]
        r = srv.wait(srv.evolve(m, pos, vel, 0.03, 1.0))
        busy = srv.stats()["busy_s"] - before
    took = r["t_done"] - r["t_start"]
    assert took > 0.001
    assert 0.5 * took < busy <= 1.01 * took + 1e-3


def test_requests_and_cancellations_during_a_cluster_launch(nb):
    """A request that arrives while only a cluster launch is under way is served beside it, and
    a cancelled integration ends with the launch."""
    rng = np.random.default_rng(7)
    m, pos, vel = np.full(3000, 1 / 3000.0), rng.standard_normal((3, 3000)), np.zeros((3, 3000))
    with nb.Server(dt_max=1.0 / 16) as srv:
        long = srv.evolve(m, pos, vel, 0.01, 64.0)
        for _ in range(5):
            f = srv.wait(srv.force(m[:100], pos[:, :100].copy(), vel[:, :100].copy(), 0.01))
            assert f["status"] == nb.NB_STATUS_DONE
        assert srv.poll(long)["status"] not in (nb.NB_STATUS_DONE, nb.NB_STATUS_ERROR)
        srv.cancel(long)
        assert srv.wait(long)["status"] == nb.NB_STATUS_CANCELLED
