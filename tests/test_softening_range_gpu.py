"""Softenings far from the system's size: self pairs, padding, units of length.

Gates are those of the other kernels (forces 1e-5, jerk 1e-4, both per
particle; VJP with split positions 2e-6 of the largest gradient), against the
oracle's FP64 pairs.
"""
import numpy as np
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


def check(pos, vel, mass, eps, pairs="default", jerk=True, vjp=True):
    n = mass.shape[0]
    cot = np.random.default_rng(n).normal(size=(n, 3))
    ra, rj, rp = oracle.forces_jerk(pos, vel, mass, eps)
    o = binding.make_opts("f64acc", positions="split", pairs=pairs)
    ws = binding.workspace(n, 1, o)
    x, v, m = dev(pos), dev(vel), dev(mass)
    acc, jk, xb = (torch.empty_like(x) for _ in range(3))
    pot, mb = torch.empty_like(m), torch.empty_like(m)
    binding.nb_forces(x, m, eps, acc, pot, ws, o)
    assert binding.nb_poll_status(ws, o) == binding.NB_OK
    assert rel_vec_err(host(acc), ra).max() <= 1e-5 and rel_err(host(pot), rp).max() <= 1e-5
    if jerk:
        binding.nb_forces_jerk(x, v, m, eps, acc, jk, pot, ws, o)
        assert binding.nb_poll_status(ws, o) == binding.NB_OK
        assert rel_vec_err(host(acc), ra).max() <= 1e-5 and rel_err(host(pot), rp).max() <= 1e-5
        assert rel_vec_err(host(jk), rj).max() <= 1e-4
    if vjp:
        rx, rm = oracle.forces_vjp(pos, mass, eps, cot, None)
        binding.nb_forces_vjp(x, m, eps, dev(cot), None, xb, mb, ws, o)
        assert binding.nb_poll_status(ws, o) == binding.NB_OK
        assert np.abs(host(xb) - rx).max() <= 2e-6 * np.abs(rx).max()
        assert np.abs(host(mb) - rm).max() <= 2e-6 * np.abs(rm).max()


@pytest.mark.parametrize("n", [301, 2047, 5001, 12289])
@pytest.mark.parametrize("where", [1e4, 1e6, 1e9])
def test_an_escaper_beside_a_small_softening(n, where):
    """eps / max|x| of 1e-12 to 1e-17: r^-3 of a particle with itself is beyond
    FP32 in units of max|x|."""
    s = ics.plummer_lognormal(n, seed=n)
    s.pos[n // 2] = (where, -0.3 * where, 0.1 * where)
    s.vel[n // 2] = (3.0, 1.0, -2.0)
    check(s.pos, s.vel, s.mass, 1e-8)


@pytest.mark.parametrize("eps", [1e-8, 1e-12, 1e-15, 1.2e-19])
def test_a_particle_at_the_origin(eps):
    """On the spot where a zero-filled pack has its padding."""
    n = 4801
    s = ics.plummer_lognormal(n, seed=5)
    s.pos[17] = 0.0
    check(s.pos, s.vel, s.mass, eps)
    check(s.pos, s.vel, s.mass, eps, pairs="symmetric")


@pytest.mark.parametrize("n", [301, 5001])
def test_two_particles_on_one_spot(n):
    """d = 0: no force, the largest potential (m / eps) and jerk (m w / eps^3)."""
    s = ics.plummer_lognormal(n, seed=n)
    s.pos[n - 1] = s.pos[3]
    check(s.pos, s.vel, s.mass, 1e-8, vjp=False)


@pytest.mark.parametrize("n,size,eps", [(301, 1e-14, 1.0), (5001, 1e-14, 1.0), (301, 1e-9, 1e6),
                                        (5001, 1e-9, 1e6), (5001, 1e12, 1e9), (5001, 1e12, 1e2),
                                        (301, 1e-6, 1e-7), (5001, 1e-6, 1e-7)])
def test_units_of_length(n, size, eps):
    s = ics.plummer_lognormal(n, seed=n)
    check(size * s.pos, s.vel, s.mass, eps)


@pytest.mark.parametrize("n", [300, 5001, 12001])
@pytest.mark.parametrize("eps", [1e-8, 0.999e-8, 1e-12, 1e-16, 1.2e-19])
def test_tiny_softening(n, eps):
    """The totals' bounds grow with eps^-2 and eps^-3; their grid must not."""
    s = ics.plummer_lognormal(n, seed=n)
    check(s.pos, s.vel, s.mass, eps)


@pytest.mark.parametrize("n", [300, 5001])
@pytest.mark.parametrize("eps", [1e-8, 0.999e-8, 1e-14, 0.999e-14, 1e-16, 1.2e-19])
def test_fp64_pairs_at_tiny_softening(n, eps):
    """Symmetric from 1e-14, direct below."""
    s = ics.plummer_lognormal(n, seed=n)
    ra, rp = oracle.forces(s.pos, s.mass, eps, 1.0)
    o = binding.make_opts("fp64")
    ws = binding.workspace(n, 1, o)
    x, m = dev(s.pos), dev(s.mass)
    acc, pot = torch.empty_like(x), torch.empty_like(m)
    binding.nb_forces(x, m, eps, acc, pot, ws, o)
    assert binding.nb_poll_status(ws, o) == binding.NB_OK
    assert rel_vec_err(host(acc), ra).max() <= 1e-12 and rel_err(host(pot), rp).max() <= 1e-12


def test_fp64_symmetric_pair_terms_over_magnitudes():
    """test_sym64_gpu's pair terms on the symmetric kernel, asked for by name:
    the reciprocal root over 69 decades."""
    n, eps = 200, 1e-10
    d = np.concatenate([[0.0], np.logspace(-9, 60, n - 1) * np.linspace(1.0, 1.9, n - 1)])
    pos = np.zeros((n, 3))
    pos[:, 0] = d
    mass = np.full(n, 1e-300)
    mass[0] = 1.0
    o = binding.make_opts("fp64", pairs="symmetric")
    ws = binding.workspace(n, 1, o)
    x, m = dev(pos), dev(mass)
    acc, pot = torch.empty_like(x), torch.empty_like(m)
    binding.nb_forces(x, m, eps, acc, pot, ws, o)
    dl = d[1:].astype(np.longdouble)
    r2 = dl * dl + np.longdouble(eps) ** 2
    ref = -dl / (r2 * np.sqrt(r2))
    big = np.abs(ref) > 2.0 ** -120 * 1.02 * n * 0.385 / eps ** 2
    assert np.abs(host(acc)[1:, 0][big] / ref[big] - 1).max() <= 2e-15
    assert np.abs(host(pot)[1:] * np.sqrt(r2) + 1)[big].max() <= 2e-15


@pytest.mark.parametrize("prec", ["kahan", "fp32"])
def test_large_system_at_tiny_softening(prec):
    """Above 24576 particles, where the adaptive path's grid has 100 bits."""
    n, eps = 66000, 1e-12
    s = ics.plummer_lognormal(n, seed=2)
    rows = np.arange(0, n, 331)
    ra, rp = oracle.forces_rows(s.pos, s.mass, eps, rows)
    o = binding.make_opts(prec)
    ws = binding.workspace(n, 1, o)
    x, m = dev(s.pos), dev(s.mass)
    acc, pot = torch.empty_like(x), torch.empty_like(m)
    binding.nb_forces(x, m, eps, acc, pot, ws, o)
    assert binding.nb_poll_status(ws, o) == binding.NB_OK
    gate = 1e-5 if prec == "kahan" else 1e-4
    assert rel_vec_err(host(acc)[rows], ra).max() <= gate
    assert rel_err(host(pot)[rows], rp).max() <= gate
