"""GPU parity of the warp-granular symmetric-pair kernels (forces, VJP,
acceleration + jerk) at the edges of their blocks, ranges and shapes, against
the oracle.

The blocks are 128 or 256 slots, j-sets 32 or 64, and the pairs of a system
are cut into one range of rotation steps per warp, so the sizes are one
particle past, at and below whole blocks, fewer blocks than warps, and both
sides of the sizes at which the shape changes (12288 forces, 24576 jerk).
Tolerances are the gates of the other kernels: forces 1e-5 (split), jerk 1e-4,
VJP with split positions 2e-6 of the largest gradient.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_02744_gb300 import api, binding, ics
from tests.gpu_util import dev, host, rel_err, rel_vec_err

pytestmark = pytest.mark.gpu

EPS = 0.01


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    oracle.build()
    binding.lib()


@pytest.mark.parametrize("prec", ["kahan", "f64acc", "fp32"])
@pytest.mark.parametrize("n", [2, 127, 129, 255, 257, 4800, 12287, 12289])
def test_forces_at_block_edges(n, prec):
    s = ics.plummer_lognormal(n, seed=n)
    ra, rp = oracle.forces(s.pos, s.mass, EPS, 1.5)
    # the single-float form against the direct kernel of the same form
    positions = "single" if prec == "fp32" else "split"
    a, p = api.forces(dev(s.pos), dev(s.mass), EPS, precision=prec, G=1.5, positions=positions,
                      pairs="symmetric")
    a2, _ = api.forces(dev(s.pos), dev(s.mass), EPS, precision=prec, G=1.5, positions=positions,
                       pairs="symmetric", with_pot=False)
    assert torch.equal(a, a2)  # the potential changes no acceleration
    if prec == "fp32":
        d, dp = api.forces(dev(s.pos), dev(s.mass), EPS, precision="f64acc", G=1.5,
                           positions="single", pairs="direct")
        ra, rp = host(d), host(dp)
    assert rel_vec_err(host(a), ra).max() <= 1e-5 and rel_err(host(p), rp).max() <= 1e-5


@pytest.mark.parametrize("n", [256, 257, 2047, 2049, 4097])
@pytest.mark.parametrize("with_pbar", [False, True])
def test_vjp_at_block_edges(n, with_pbar):
    s = ics.plummer_lognormal(n, seed=n)
    rng = np.random.default_rng(n)
    abar = rng.normal(size=(n, 3))
    pbar = rng.normal(size=n) if with_pbar else None
    rx, rm = oracle.forces_vjp(s.pos, s.mass, EPS, abar, pbar)
    o = binding.make_opts("f64acc", positions="split")
    ws = binding.workspace(n, 1, o)
    pos, mass, ab = dev(s.pos), dev(s.mass), dev(abar)
    pb = None if pbar is None else dev(pbar)
    out = []
    for _ in range(2):  # the second call starts from the words the first one left
        xb = torch.empty((n, 3), dtype=torch.float64, device="cuda")
        mb = torch.empty(n, dtype=torch.float64, device="cuda")
        binding.nb_forces_vjp(pos, mass, EPS, ab, pb, xb, mb, ws, o)
        out.append((xb, mb))
    assert binding.nb_poll_status(ws, o) == binding.NB_OK
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert np.abs(host(out[0][0]) - rx).max() <= 2e-6 * np.abs(rx).max()
    assert np.abs(host(out[0][1]) - rm).max() <= 2e-6 * np.abs(rm).max()


@pytest.mark.parametrize("n", [256, 257, 3000, 12289])
def test_jerk_at_block_edges(n):
    s = ics.plummer_lognormal(n, seed=n)
    ra, rj, rp = oracle.forces_jerk(s.pos, s.vel, s.mass, EPS)
    o = binding.make_opts("kahan")
    ws = binding.workspace(n, 1, o)
    pos, vel, mass = dev(s.pos), dev(s.vel), dev(s.mass)
    acc, jerk = torch.empty_like(pos), torch.empty_like(pos)
    pot = torch.empty_like(mass)
    for with_pot in (False, True):
        binding.nb_forces_jerk(pos, vel, mass, EPS, acc, jerk, pot if with_pot else None, ws, o)
        assert binding.nb_poll_status(ws, o) == binding.NB_OK
        assert rel_vec_err(host(acc), ra).max() <= 1e-5
        assert rel_vec_err(host(jerk), rj).max() <= 1e-4
    assert rel_err(host(pot), rp).max() <= 1e-5


@pytest.mark.parametrize("eps", [1e-5, 1e-8])
def test_small_softening(eps):
    """The a-priori bounds that place the fixed-point grid grow with eps^-2
    (forces) and eps^-3 (VJP, jerk): at a softening far below the closest pair
    the results still meet the gates."""
    n = 5000
    s = ics.plummer_lognormal(n, seed=21)
    ra, rj, rp = oracle.forces_jerk(s.pos, s.vel, s.mass, eps)
    cot = np.random.default_rng(21).normal(size=(n, 3))
    rx, rm = oracle.forces_vjp(s.pos, s.mass, eps, cot, None)
    o = binding.make_opts("f64acc", positions="split")
    ws = binding.workspace(n, 1, o)
    pos, vel, mass = dev(s.pos), dev(s.vel), dev(s.mass)
    acc, jerk, xb = (torch.empty_like(pos) for _ in range(3))
    pot, mb = torch.empty_like(mass), torch.empty_like(mass)
    binding.nb_forces(pos, mass, eps, acc, pot, ws, o)
    assert rel_vec_err(host(acc), ra).max() <= 1e-5 and rel_err(host(pot), rp).max() <= 1e-5
    binding.nb_forces_jerk(pos, vel, mass, eps, acc, jerk, pot, ws, o)
    assert rel_vec_err(host(acc), ra).max() <= 1e-5
    assert rel_vec_err(host(jerk), rj).max() <= 1e-4
    binding.nb_forces_vjp(pos, mass, eps, dev(cot), None, xb, mb, ws, o)
    assert binding.nb_poll_status(ws, o) == binding.NB_OK
    assert np.abs(host(xb) - rx).max() <= 2e-6 * np.abs(rx).max()
    assert np.abs(host(mb) - rm).max() <= 2e-6 * np.abs(rm).max()


def test_one_workspace_serves_every_kernel():
    """Forces, VJP and jerk of one system in turn on one workspace: each
    leaves its totals and maxima cleared for the next."""
    n = 6000
    s = ics.plummer_lognormal(n, seed=3)
    o = binding.make_opts("f64acc", positions="split")
    pos, vel, mass = dev(s.pos), dev(s.vel), dev(s.mass)
    cot = dev(np.random.default_rng(3).normal(size=(n, 3)))

    def run(ws):
        acc, jerk, xb = (torch.empty_like(pos) for _ in range(3))
        pot, mb = torch.empty_like(mass), torch.empty_like(mass)
        binding.nb_forces(pos, mass, EPS, acc, pot, ws[0], o)
        out = [acc.clone(), pot.clone()]
        binding.nb_forces_vjp(pos, mass, EPS, cot, None, xb, mb, ws[1], o)
        binding.nb_forces_jerk(pos, vel, mass, EPS, acc, jerk, None, ws[2], o)
        return out + [xb, mb, acc, jerk]

    shared = binding.workspace(n, 1, o)
    want = run([binding.workspace(n, 1, o) for _ in range(3)])
    for _ in range(2):
        for a, b in zip(run([shared] * 3), want):
            assert torch.equal(a, b)
    assert binding.nb_poll_status(shared, o) == binding.NB_OK
