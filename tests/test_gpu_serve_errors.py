"""Failures of the request loop's integrations in their cluster launches."""
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
