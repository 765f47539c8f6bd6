"""The first force evaluation of a handle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ni", [(2500, 2500), (8192, 8192), (20011, 3000), (20011, 5000),
                                  (65536, 1531)])
def test_first_short_evaluation_allocates_no_partials(nb, n, ni):
    """A short evaluation whose j-splits' partials take over 1 MB (a mapping of its own, which
    takes the device longer than the split saves) finds room for them in the handle. Watched by
    the device's free memory, which only such mappings change."""
    import torch
    rng = np.random.default_rng(3)
    m, x, v = np.full(n, 1.0 / n), rng.standard_normal((n, 3)), rng.standard_normal((n, 3))
    out = torch.empty((7, ni), dtype=torch.float64, device="cuda")
    p = out.data_ptr()
    idx = torch.arange(ni, dtype=torch.int32, device="cuda")
    for rep in range(2):  # the first pass loads the kernels
        with nb.System(m, x, v, variant="f32ds", eps=0.01) as sy:
            sy.predict(0.0)
            nsplit = nb.nb_plan_for(sy.h, ni)[2]
            assert nsplit * 7 * ni * 8 > 1 << 20
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info(0)[0]
            nb.nb_force_dev(sy.h, idx.data_ptr(), ni, p, p + 24 * ni, p + 48 * ni)
            used = free - torch.cuda.mem_get_info(0)[0]
        if rep:
            assert used < 1 << 20
