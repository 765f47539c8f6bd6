"""The pair kernels take the bare SFU reciprocal square root where eps^2 >= FLT_MIN (every
r^2 + eps^2 is then a normal FP32 number) and rsqrtf below. Around that line eps^2 is far
under half an ulp of every r^2 here (r > 1e-6), so two softenings on either side of it round
every r^2 + eps^2 alike (up where dx^2 alone would be a tie: eps = 0 is not in the comparison
for that reason) and must give the same bits, on every kernel and at ragged sizes; ordinary
softenings and eps = 0 are gated against the oracle elsewhere."""
import numpy as np
import pytest

from paper_1409_5474_gb300 import ic

pytestmark = pytest.mark.gpu

FLT_MIN = 2.0 ** -126
EPS = {"general": 1.0e-19, "soft": 1.1e-19}  # eps^2 = 1.0e-38 and 1.21e-38
assert np.float32(EPS["general"] ** 2) < FLT_MIN <= np.float32(EPS["soft"] ** 2)

# plan-table entries (kind, warp rows, splits) that reach each kernel
PLANS = {"tile1": (0, 1, 3), "tile4": (0, 4, 2), "tile8": (0, 8, 5), "wgrp": (1, 1, 3),
         "tiny": (2, 1, 1)}


def _force(nb, p, eps, variant, plan, idx, order=4):
    with nb.System(p.m, p.pos, p.vel, variant=variant, eps=eps, order=order, device=0) as s:
        if plan is not None:
            nb.nb_set_plan_table(s.h, [plan] * 32)
        s.predict(0.0)
        return s.force_snap(idx) if order == 6 else s.force(idx)


@pytest.mark.parametrize("variant", ["f32ds", "f32"])
@pytest.mark.parametrize("plan", sorted(PLANS))
@pytest.mark.parametrize("n", [255, 1025, 2304])
def test_bits_across_the_line(nb, variant, plan, n):
    p = ic.plummer(n, 31 + n, masses="lognormal")
    idx = None if plan != "tiny" else np.arange(0, n, n // 3, dtype=np.int32)
    got = [_force(nb, p, eps, variant, PLANS[plan], idx) for eps in EPS.values()]
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("nwj", [1, 2, 4, 8])
def test_bits_across_the_line_order6(nb, nwj):
    p = ic.plummer(901, 5, masses="lognormal")
    got = [_force(nb, p, eps, "f32ds", (0, nwj, 2), None, order=6) for eps in EPS.values()]
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


def test_bits_across_the_line_batch(nb):
    systems = [ic.plummer(n, n) for n in (16, 130, 257, 700)]
    got = []
    for eps in EPS.values():
        with nb.Batch(systems, [eps] * 4, 1.0 / 4096, device=0) as b:
            b.step(2)
            got.append(b.get()[:2])
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("order", [4, 6])
def test_bits_across_the_line_block_steps(nb, order):
    """Small and mid-size due sets of the fused kernels and the planned ones."""
    p = ic.plummer(3000, 8)
    got = []
    for eps in EPS.values():
        with nb.System(p.m, p.pos, p.vel, variant="f32ds", eps=eps, eta=0.02, order=order,
                       device=0) as s:
            s.step(1.0 / 512)
            st = s.state()
            got.append((st["pos"], st["vel"]))
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
