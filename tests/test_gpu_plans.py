"""Force plans at the edges of their rules: the tiny-set kernel's j-set limit, one and two
i-particles per lane, every way the split reduction is launched (one or eight threads per
output, ragged groups of splits), against the oracle with the gates of the force tests."""
import numpy as np
import pytest

import oracle
from paper_1409_5474_gb300 import ic
from tests.test_gpu_force import _gate

pytestmark = pytest.mark.gpu


def _one(nb, variant, p, eps, idx, plan=None, kind=None):
    with nb.System(p.m, p.pos, p.vel, variant=variant, eps=eps, device=0) as s:
        if plan is not None:
            nb.nb_set_plan_table(s.h, [plan] * 32)
        s.predict(0.0)
        if kind is not None:
            assert nb.nb_plan_for(s.h, len(idx))[0] == kind
        got = s.force(idx)
    ref = oracle.force(p.m, p.pos, p.vel, eps * eps, idx=idx)
    _gate(variant, *got, *ref, tag=(p.n, len(idx), plan))


@pytest.mark.parametrize("variant", ["f32ds", "f32"])
@pytest.mark.parametrize("n_i", [1, 32, 33, 700])
@pytest.mark.parametrize("nsplit", [1, 2, 8, 9, 17, 18])
def test_splits(nb, variant, n_i, nsplit):
    p = ic.plummer(4500, 3, masses="lognormal")  # 17 full tiles and a ragged one
    idx = np.sort(np.random.default_rng(n_i).permutation(4500)[:n_i]).astype(np.int32)
    _one(nb, variant, p, 1e-3, idx, plan=(0, 8, nsplit))


@pytest.mark.parametrize("n_i", [1, 4, 31, 33, 200])
@pytest.mark.parametrize("plan", [(0, 1, 1), (0, 1, 7), (0, 1, 8), (0, 1, 63), (1, 1, 1), (1, 1, 9)])
def test_splits_fp64(nb, plan, n_i):
    p = ic.plummer(999, 5, masses="lognormal")  # 62 units of 16 j and one of 7
    idx = np.random.default_rng(n_i).integers(0, 999, n_i).astype(np.int32)
    _one(nb, "f64", p, 1e-3, idx, plan=plan)


@pytest.mark.parametrize("n,n_i,kind", [(65536, 4, 2), (65536, 5, 0), (65537, 5, 2), (65537, 8, 2),
                                        (65537, 9, 0)])
def test_tiny_sets(nb, n, n_i, kind):
    """Up to four members, up to eight on a j-set over 65536 (two passes); then tiles."""
    p = ic.plummer(n, 4, masses="lognormal")
    idx = np.linspace(0, n - 1, n_i).astype(np.int32)
    _one(nb, "f32ds", p, 1e-3, idx, kind=kind)
