"""GPU parity of the small-system kernel (whole rows per CTA) against the
oracle: fewer particles than SMs, ragged row groups and j-sets, and its
one-kernel step loop with both packed buffers."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_02744_gb300 import api, binding, ics
from tests.gpu_util import dev, host, rel_err, rel_vec_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    oracle.build()
    binding.lib()


@pytest.mark.parametrize("prec", ["kahan", "f64acc", "fp32"])
@pytest.mark.parametrize("n", [1, 2, 63, 65, 151, 153, 607, 1025, 4799])
def test_small_forces_match_oracle(n, prec):
    s = ics.plummer_lognormal(n, seed=n)
    ra, rp = oracle.forces(s.pos, s.mass, 0.02, 2.0)
    a, p = api.forces(dev(s.pos), dev(s.mass), 0.02, precision=prec, G=2.0, positions="split")
    assert rel_vec_err(host(a), ra).max() <= 1e-5 and rel_err(host(p), rp).max() <= 1e-5
    if n == 1:
        assert torch.all(a == 0.0) and torch.all(p == 0.0)


@pytest.mark.parametrize("n", [3, 100, 2049])
@pytest.mark.parametrize("nsteps", [1, 2, 7])
def test_small_step_loop_matches_oracle(n, nsteps):
    # two calls: the first starts without accelerations, the second reuses them
    s = ics.plummer(n, seed=n)
    eps, h = 0.02, 1e-3
    g = api.System(s.pos, s.vel, s.mass, eps)
    g.step(h, nsteps)
    g.step(h, nsteps)
    assert g.poll() == binding.NB_OK
    xo, vo, ao, po = oracle.kdk(s.pos, s.vel, s.mass, eps, h, 2 * nsteps)
    assert np.abs(host(g.pos) - xo).max() <= 1e-5 * np.abs(xo - s.pos).max()
    assert np.abs(host(g.vel) - vo).max() <= 1e-5 * np.abs(vo - s.vel).max()
    assert rel_vec_err(host(g.acc), ao).max() <= 1e-5
    assert rel_err(host(g.pot), po).max() <= 1e-5
