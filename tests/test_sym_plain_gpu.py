"""Forces with one displacement form for every pair on both sides of the size
where the symmetric kernel changes (38912), and the step loop above it."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_02744_gb300 import api, binding, ics
from tests.gpu_util import dev, host, rel_err, rel_vec_err

pytestmark = pytest.mark.gpu

EPS = 5e-3


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    oracle.build()
    binding.lib()


@pytest.mark.parametrize("n", [38911, 38912, 40961])
@pytest.mark.parametrize("prec,positions", [("fp32", "default"), ("kahan", "split"),
                                            ("f64acc", "split"), ("f64acc", "single")])
def test_forces_around_the_change(n, prec, positions):
    s = ics.plummer_lognormal(n, seed=n)
    x, m = dev(s.pos), dev(s.mass)
    a, p = api.forces(x, m, EPS, precision=prec, positions=positions)
    a2, _ = api.forces(x, m, EPS, precision=prec, positions=positions, with_pot=False)
    assert torch.equal(a, a2)
    if positions == "split":
        rows = np.arange(0, n, 97)
        ra, rp = oracle.forces_rows(s.pos, s.mass, EPS, rows)
        a, p = host(a)[rows], host(p)[rows]
    else:  # the same rounded positions by every ordered pair
        d, dp = api.forces(x, m, EPS, precision="f64acc", positions="single", pairs="direct")
        a, p, ra, rp = host(a), host(p), host(d), host(dp)
    gate = 1e-4 if prec == "fp32" else 1e-5
    assert rel_vec_err(a, ra).max() <= gate and rel_err(p, rp).max() <= gate


@pytest.mark.parametrize("prec,positions", [("fp32", "default"), ("f64acc", "split")])
@pytest.mark.parametrize("valid", [False, True])
def test_step_loop_equals_single_steps(prec, positions, valid):
    """Ranges once per call and kick, drift and pack in the fold, against one
    call per step: the same sums in the same order, kicks rounded alike but for
    the fused multiply-adds of two kernels (1e-15 of the step's change)."""
    n, h, steps = 38913, 1e-4, 3
    s = ics.plummer_lognormal(n, seed=3)
    loop, single = (api.System(s.pos, s.vel, s.mass, EPS, precision=prec, positions=positions)
                    for _ in range(2))
    if valid:
        loop.forces()
        single.forces()
    loop.step(h, steps)
    for _ in range(steps):
        single.step(h, 1)
    assert loop.poll() == binding.NB_OK and single.poll() == binding.NB_OK
    assert np.abs(host(loop.vel) - host(single.vel)).max() <= 1e-13
    assert np.abs(host(loop.pos) - host(single.pos)).max() <= 1e-13
    assert rel_vec_err(host(loop.acc), host(single.acc)).max() <= 1e-5
    assert rel_err(host(loop.pot), host(single.pot)).max() <= 1e-5
