"""Batched systems above 1024 particles: their j-range is taken in parts, whose sums are added
in one order wherever the parts run, so a system's bits depend on the system alone."""
import numpy as np
import pytest

from paper_1409_5474_gb300 import ic

pytestmark = pytest.mark.gpu

DT = 1.0 / 512


def _smallest_budget(nb, sizes, variant):
    """The least budget_bytes that nb_batch_create accepts: the state, no partials."""
    lo, hi = 1, 1 << 30
    while lo < hi:
        mid = (lo + hi) // 2
        cfg = nb.nb_config_default(variant=variant, device=0, budget_bytes=mid)
        try:
            nb.nb_batch_destroy(nb.nb_batch_create(cfg, sizes, [0.05] * len(sizes), DT))
            hi = mid
        except nb.NBodyError as e:
            assert e.status == nb.NB_ERR_BUDGET
            lo = mid + 1
    return lo


def _run(nb, systems, tune=False, **cfg):
    eps = np.full(len(systems), 0.05)
    with nb.Batch(systems, eps, DT, device=0, **cfg) as b:
        if tune:
            b.autotune()
        b.step(3)
        pos, vel, _ = b.get()
        return [np.concatenate([b.system(s, pos), b.system(s, vel)]) for s in range(len(systems))]


@pytest.mark.parametrize("variant", ["f32ds", "f32"])
def test_bits_depend_on_the_system_alone(nb, variant):
    sizes = [1024, 1025, 1500, 2049, 4096, 5000]
    systems = [ic.plummer(n, 70 + k) for k, n in enumerate(sizes)]
    mix = _run(nb, systems, variant=variant)
    tight = _run(nb, systems, variant=variant, budget_bytes=_smallest_budget(nb, sizes, variant))
    tuned = _run(nb, systems, tune=True, variant=variant)
    for s, p in enumerate(systems):
        alone = _run(nb, [p], variant=variant)[0]
        np.testing.assert_array_equal(mix[s], alone)
        np.testing.assert_array_equal(tight[s], alone)
        np.testing.assert_array_equal(tuned[s], alone)


def test_partials_of_a_large_system_are_bounded(nb):
    """262144 particles: 272 bytes of state and 4 x 56 of partials each, 130 MB; the allocator
    hands out whole blocks of a few MB and the launches' own buffers come on top. Parts of
    1024 would take 3.8 GB."""
    import torch
    rng = np.random.default_rng(2)
    n = 262144
    m, pos, vel = np.full(n, 1.0 / n), rng.standard_normal((3, n)), rng.standard_normal((3, n))
    cfg = nb.nb_config_default(variant="f32ds", device=0)
    b = nb.nb_batch_create(cfg, [64], [0.05], DT)
    nb.nb_batch_set(b, m[:64], pos[:, :64].copy(), vel[:, :64].copy())
    nb.nb_batch_step(b, 1)  # the module is loaded
    nb.nb_batch_destroy(b)
    free = torch.cuda.mem_get_info(0)[0]
    b = nb.nb_batch_create(cfg, [n], [0.05], DT)
    nb.nb_batch_set(b, m, pos, vel)
    nb.nb_batch_step(b, 1)
    used = free - torch.cuda.mem_get_info(0)[0]
    nb.nb_batch_destroy(b)
    assert used < 192 << 20


def test_autotune_between_steps(nb):
    """The autotuner rebuilds the lists after a step was captured: the next step is captured anew."""
    systems = [ic.plummer(n, 80 + k) for k, n in enumerate((70, 900, 1100, 2500))]
    eps = np.full(4, 0.05)
    got = []
    for tune in (False, True):
        with nb.Batch(systems, eps, DT, variant="f32ds", device=0) as b:
            b.step(2)
            if tune:
                b.autotune()
            b.step(2)
            got.append(b.get()[:2])
    np.testing.assert_array_equal(got[0], got[1])
