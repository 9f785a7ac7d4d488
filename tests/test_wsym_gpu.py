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
