"""GPU parity of the FP64 symmetric-pair kernel at the edges of its blocks and
ranges, and of its reciprocal square root over many magnitudes."""
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


@pytest.mark.parametrize("n", [63, 64, 65, 127, 1000, 4097])
@pytest.mark.parametrize("eps", [0.01, 1e-7])
def test_fp64_forces_match_oracle(n, eps):
    s = ics.plummer_lognormal(n, seed=n)
    ra, rp = oracle.forces(s.pos, s.mass, eps, 2.0)
    a, p = api.forces(dev(s.pos), dev(s.mass), eps, precision="fp64", G=2.0)
    a2, _ = api.forces(dev(s.pos), dev(s.mass), eps, precision="fp64", G=2.0, with_pot=False)
    assert torch.equal(a, a2)
    assert rel_vec_err(host(a), ra).max() <= 1e-12 and rel_err(host(p), rp).max() <= 1e-12


def test_fp64_pair_term_over_magnitudes():
    """199 test particles (mass 1e-300) around a unit mass at distances from
    1e-9 to 1e60: each acceleration is one pair term.  At most ~8 roundings of
    2^-53 and three times the reciprocal root's error: 2e-15."""
    n, eps = 200, 1e-10
    d = np.concatenate([[0.0], np.logspace(-9, 60, n - 1) * np.linspace(1.0, 1.9, n - 1)])
    pos = np.zeros((n, 3))
    pos[:, 0] = d
    mass = np.full(n, 1e-300)
    mass[0] = 1.0
    a, p = api.forces(dev(pos), dev(mass), eps, precision="fp64")
    dl = d[1:].astype(np.longdouble)
    r2 = dl * dl + np.longdouble(eps) ** 2
    ref = -dl / (r2 * np.sqrt(r2))
    # the totals' grid is at most 2^-173 of the bound on them (nbody.h): rounding
    # to it stays below 2^-53 of values above 2^-120 of the bound
    big = np.abs(ref) > 2.0 ** -120 * 1.02 * n * 0.385 / eps ** 2
    assert big.sum() > 40
    assert np.abs(host(a)[1:, 0][big] / ref[big] - 1).max() <= 2e-15
    assert np.abs(host(p)[1:] * np.sqrt(r2) + 1)[big].max() <= 2e-15
    assert np.all(np.isfinite(host(a))) and np.all(np.isfinite(host(p)))


@pytest.mark.parametrize("nsteps", [1, 3])
def test_fp64_step_loop_matches_oracle(nsteps):
    n, eps, h = 300, 0.02, 1e-3
    s = ics.plummer(n, seed=n)
    g = api.System(s.pos, s.vel, s.mass, eps, precision="fp64")
    g.step(h, nsteps)
    g.step(h, nsteps)
    assert g.poll() == binding.NB_OK
    xo, vo, ao, po = oracle.kdk(s.pos, s.vel, s.mass, eps, h, 2 * nsteps)
    assert np.abs(host(g.pos) - xo).max() <= 1e-13 * np.abs(xo).max()
    assert np.abs(host(g.vel) - vo).max() <= 1e-13 * np.abs(vo).max()
    assert rel_vec_err(host(g.acc), ao).max() <= 1e-11
    assert rel_err(host(g.pot), po).max() <= 1e-12
