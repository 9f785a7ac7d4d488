"""The adaptive symmetric path's step loop (fold, kicks, drift, pack and boxes
in one kernel between re-sorts) at ragged sizes and across a re-sort, against
the same steps made one call at a time, each of which sorts and packs afresh."""
import numpy as np
import pytest
import torch

from paper_2605_02744_gb300 import api, binding, ics
from tests.gpu_util import host, rel_vec_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    binding.lib()


@pytest.mark.parametrize("n", [1, 255, 2047, 2049, 6500])
@pytest.mark.parametrize("valid", [False, True])
def test_step_loop_equals_single_steps(n, valid):
    s = ics.plummer_lognormal(n, seed=n)
    eps, h, steps = 5e-3, 1e-4, 18
    opts = dict(precision="f64acc", positions="adaptive", pairs="symmetric")
    loop, single = (api.System(s.pos, s.vel, s.mass, eps, **opts) for _ in range(2))
    if valid:
        loop.forces()
        single.forces()
    loop.step(h, steps)
    for _ in range(steps):
        single.step(h, 1)
    assert loop.poll() == binding.NB_OK and single.poll() == binding.NB_OK
    # the orders differ (re-sorted after 16 steps against every step): rounding
    # of FP32 sums only, 1e-5 of an acceleration, dt^2 and dt times that here
    if n > 1:
        assert rel_vec_err(host(loop.acc), host(single.acc)).max() <= 2e-5
    dx = max(np.abs(host(single.pos) - s.pos).max(), 1e-300)
    assert np.abs(host(loop.pos) - host(single.pos)).max() <= 1e-6 * dx
    assert torch.all(torch.isfinite(loop.pot))
