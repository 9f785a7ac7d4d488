"""Inputs that are not finite, or far from 1, on the paths that combine partial
sums in fixed point: a NaN or infinite input shows in the outputs and in the
status word, the next call on the same workspace is clean, and FP64 pairs take
masses outside the range of FP32."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_02744_gb300 import binding, ics
from tests.gpu_util import dev, host, rel_err, rel_vec_err

pytestmark = pytest.mark.gpu

EPS = 0.02


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    oracle.build()
    binding.lib()


def _calls(n, prec, pos, vel, mass, cot, ws, o):
    acc, jerk, xb = (torch.zeros_like(pos) for _ in range(3))
    pot, mb = torch.zeros_like(mass), torch.zeros_like(mass)
    yield "forces", lambda: binding.nb_forces(pos, mass, EPS, acc, pot, ws, o), (acc, pot)
    if prec != "fp64":
        yield "vjp", lambda: binding.nb_forces_vjp(pos, mass, EPS, cot, None, xb, mb, ws, o), (xb, mb)
        yield "jerk", lambda: binding.nb_forces_jerk(pos, vel, mass, EPS, acc, jerk, None, ws, o), \
            (acc, jerk)


@pytest.mark.parametrize("n,prec", [(700, "f64acc"), (5000, "f64acc"), (700, "fp64")])
@pytest.mark.parametrize("where", ["pos", "mass"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_not_finite_inputs_show(n, prec, where, value):
    s = ics.plummer(n, seed=4)
    o = binding.make_opts(prec)
    ws = binding.workspace(n, 1, o)
    pos, vel, mass = dev(s.pos), dev(s.vel), dev(s.mass)
    cot = dev(np.random.default_rng(4).normal(size=(n, 3)))
    clean = {name: (call(), [t.clone() for t in out])[1]
             for name, call, out in _calls(n, prec, pos, vel, mass, cot, ws, o)}
    assert binding.nb_poll_status(ws, o) == binding.NB_OK
    bad_pos, bad_mass = pos.clone(), mass.clone()
    if where == "pos":
        bad_pos[17, 1] = value
    else:
        bad_mass[17] = value
    for name, call, out in _calls(n, prec, bad_pos, vel, bad_mass, cot, ws, o):
        call()
        assert binding.nb_poll_status(ws, o) == binding.NB_ERR_NONFINITE, name
        others = torch.arange(n, device="cuda") != 17
        if where == "mass" and name == "vjp":
            continue  # the mass gradient does not depend on the masses
        if value != value:
            assert not torch.isfinite(out[0][others]).any(), name
    for name, call, out in _calls(n, prec, pos, vel, mass, cot, ws, o):
        call()
        for a, b in zip(out, clean[name]):
            assert torch.equal(a, b), name
    assert binding.nb_poll_status(ws, o) == binding.NB_OK


@pytest.mark.parametrize("scale", [1e45, 1e-60])
def test_fp64_masses_outside_the_fp32_range(scale):
    n = 300
    s = ics.plummer_lognormal(n, seed=5)
    o = binding.make_opts("fp64")
    ws = binding.workspace(n, 1, o)
    acc, pot = torch.empty((n, 3), dtype=torch.float64, device="cuda"), dev(s.mass).clone()
    binding.nb_forces(dev(s.pos), dev(s.mass * scale), EPS, acc, pot, ws, o)
    assert binding.nb_poll_status(ws, o) == binding.NB_OK
    ra, rp = oracle.forces(s.pos, s.mass, EPS)
    assert rel_vec_err(host(acc) / scale, ra).max() <= 1e-12
    assert rel_err(host(pot) / scale, rp).max() <= 1e-12


@pytest.mark.parametrize("length,mass_unit", [(3e12, 2e30), (1e-9, 1e-20), (1e15, 1e-3)])
def test_units_far_from_one(length, mass_unit):
    """Systems in units where r^-3 or products of masses and cotangents leave
    the range of FP32 give the scaled results of the same system in units of
    order one."""
    n = 5000
    s = ics.plummer_lognormal(n, seed=6)
    o = binding.make_opts("f64acc", positions="split")
    ws = binding.workspace(n, 1, o)
    cot = np.random.default_rng(6).normal(size=(n, 3)) * 1e-12
    pbar = np.random.default_rng(7).normal(size=n) * 1e-12 / length
    ra, rj, rp = oracle.forces_jerk(s.pos, s.vel, s.mass, EPS)
    rx, rm = oracle.forces_vjp(s.pos, s.mass, EPS, cot, pbar * length)
    pos, vel, mass = dev(s.pos * length), dev(s.vel), dev(s.mass * mass_unit)
    acc, jerk, xb = (torch.empty_like(pos) for _ in range(3))
    pot, mb = torch.empty_like(mass), torch.empty_like(mass)
    ka, kp = mass_unit / length ** 2, mass_unit / length
    binding.nb_forces(pos, mass, EPS * length, acc, pot, ws, o)
    assert rel_vec_err(host(acc) / ka, ra).max() <= 1e-5
    assert rel_err(host(pot) / kp, rp).max() <= 1e-5
    binding.nb_forces_jerk(pos, vel, mass, EPS * length, acc, jerk, pot, ws, o)
    assert rel_vec_err(host(acc) / ka, ra).max() <= 1e-5
    assert rel_vec_err(host(jerk) / (ka / length), rj).max() <= 1e-4
    binding.nb_forces_vjp(pos, mass, EPS * length, dev(cot), dev(pbar), xb, mb, ws, o)
    assert binding.nb_poll_status(ws, o) == binding.NB_OK
    assert np.abs(host(xb) / (ka / length) - rx).max() <= 2e-6 * np.abs(rx).max()
    assert np.abs(host(mb) * length ** 2 - rm).max() <= 2e-6 * np.abs(rm).max()
