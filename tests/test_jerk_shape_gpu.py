"""Acceleration + jerk on both sides of the size where the symmetric kernel's
shape changes (9216)."""
import pytest
import torch

import oracle
from paper_2605_02744_gb300 import binding, ics
from tests.gpu_util import dev, host, rel_err, rel_vec_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    oracle.build()
    binding.lib()


@pytest.mark.parametrize("prec", ["kahan", "f64acc"])
@pytest.mark.parametrize("n", [9215, 9216, 9217])
def test_jerk_around_the_change(n, prec):
    s = ics.plummer_lognormal(n, seed=n)
    eps = 0.01
    ra, rj, rp = oracle.forces_jerk(s.pos, s.vel, s.mass, eps)
    o = binding.make_opts(prec)
    ws = binding.workspace(n, 1, o)
    pos, vel, mass = dev(s.pos), dev(s.vel), dev(s.mass)
    acc, jerk, pot = torch.empty_like(pos), torch.empty_like(pos), torch.empty_like(mass)
    binding.nb_forces_jerk(pos, vel, mass, eps, acc, jerk, pot, ws, o)
    assert binding.nb_poll_status(ws, o) == binding.NB_OK
    assert rel_vec_err(host(acc), ra).max() <= 1e-5 and rel_err(host(pot), rp).max() <= 1e-5
    assert rel_vec_err(host(jerk), rj).max() <= 1e-4
