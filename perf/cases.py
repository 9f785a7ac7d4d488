"""Performance cases of the direct N-body library: what its users run, by size.

Each case is one call (or one short loop) through the package's public entry
points on inputs from ``paper_2605_02744_gb300.ics``, the generators of the
tests and of the benchmark:

* ``step``      a user's integration: ``api.System.step`` (kick-drift-kick),
                optionally replayed as a CUDA graph and optionally followed by
                ``System.energy`` as the benchmark's step is.
* ``batched``   ``api.System.step`` over many independent clusters.
* ``hermite``   the fourth-order Hermite predictor-corrector around the
                acceleration + jerk evaluation (``binding.nb_hermite4``).
* ``adjoint``   a training step: ``adjoint.simulate`` inside a torch program
                whose parameters are float32 (torch's default), loss and
                gradients by autograd.
* ``labels``    accelerations and potentials of a snapshot under the FP32
                policy (``api.forces``), kept in float32 as labels of a learned
                force model.
* ``reference`` accelerations and potentials from FP64 pairs (``api.forces``),
                the grade that adjoint targets and validation runs use.

An integration returns its phase-space state (positions and velocities, FP64)
and the energies where it asked for them; the accelerations that stay in the
state are the integrator's own cache for the next call.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_02744_gb300 import adjoint, api, binding, ics

DEV = "cuda"


def listed():
    return [
        # The smallest integration of the tests: launch latency, 20 short steps.
        {"name": "step_1024", "kind": "step", "n": 1024, "masses": "equal", "eps": 0.01, "dt": 1e-3,
         "nsteps": 20, "precision": "f64acc", "graph": False, "energy": False},
        # A small system in a replayed CUDA graph, one particle short of a power of two.
        {"name": "step_4095_graph", "kind": "step", "n": 4095, "masses": "equal", "eps": 0.01,
         "dt": 1e-3, "nsteps": 20, "precision": "kahan", "graph": True, "energy": False},
        # The forward pass of the adjoint workload: the middle of the direct kernel's range.
        {"name": "step_16384", "kind": "step", "n": 16384, "masses": "equal", "eps": 5e-3,
         "dt": 1e-3, "nsteps": 10, "precision": "f64acc", "graph": False, "energy": False},
        # Ten steps of the 65536-particle log-normal mass workload.
        {"name": "step_65536_lognormal", "kind": "step", "n": 65536, "masses": "lognormal",
         "eps": 1e-3, "dt": 1e-4, "nsteps": 10, "precision": "f64acc", "graph": False,
         "energy": False},
        # The benchmark's step: one step of the 2^20 Plummer sphere and its energies.
        {"name": "step_1048576", "kind": "step", "n": 1048576, "masses": "equal", "eps": 1e-3,
         "dt": 1e-4, "nsteps": 1, "precision": "kahan", "graph": False, "energy": True},
        # The batched workload: 512 clusters of 64 to 8192 particles.
        {"name": "batched_512", "kind": "batched", "b": 512, "nmin": 64, "nmax": 8192, "eps": 0.01,
         "dt": 1e-3, "nsteps": 10, "precision": "f64acc"},
        # An ordinary Hermite run, with an odd size.
        {"name": "hermite_32769", "kind": "hermite", "n": 32769, "masses": "lognormal", "eps": 1e-3,
         "dt": 1e-4, "nsteps": 3, "precision": "f64acc"},
        # The paper's benchmark size (409600 particles), one Hermite step a call.
        {"name": "hermite_409600", "kind": "hermite", "n": 409600, "masses": "equal", "eps": 1e-3,
         "dt": 1e-4, "nsteps": 1, "precision": "kahan"},
        # A training step at the adjoint workload's size, time-reversed backward pass.
        {"name": "adjoint_16384", "kind": "adjoint", "n": 16384, "masses": "equal", "eps": 5e-3,
         "dt": 1e-3, "nsteps": 20, "segment": 10, "mode": "reverse", "precision": "f64acc"},
        # A small training step that recomputes each segment from its checkpoint.
        {"name": "adjoint_2047", "kind": "adjoint", "n": 2047, "masses": "equal", "eps": 5e-3,
         "dt": 1e-3, "nsteps": 20, "segment": 10, "mode": "recompute", "precision": "f64acc"},
        # Labels of one snapshot of the tests' odd size.
        {"name": "labels_20001", "kind": "labels", "n": 20001, "masses": "lognormal", "eps": 0.01,
         "precision": "fp32"},
        # An FP64-pair evaluation at the adjoint workload's size.
        {"name": "reference_16384", "kind": "reference", "n": 16384, "masses": "equal", "eps": 5e-3,
         "precision": "fp64"},
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi]: odd, round and in between."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batched", "hermite", "adjoint", "labels",
                       "reference"])
    masses = rng.choice(["equal", "lognormal"])
    eps = rng.choice([0.02, 0.01, 5e-3, 1e-3])
    if kind == "step":
        n = _size(rng, 256, 400000)
        # at most ~1e11 interactions a pass
        nsteps = max(1, min(rng.randint(1, 20), int(1e11 / (float(n) * n))))
        return {"kind": kind, "n": n, "masses": masses, "eps": eps,
                "dt": 1e-4 if eps < 0.01 else 5e-4, "nsteps": nsteps,
                "precision": rng.choice(["f64acc", "kahan"]), "graph": rng.random() < 0.25,
                "energy": n >= 65536 and rng.random() < 0.5}
    if kind == "batched":
        nmin = _size(rng, 64, 512)
        return {"kind": kind, "b": _size(rng, 4, 512), "nmin": nmin,
                "nmax": _size(rng, 2 * nmin, 8192), "eps": rng.choice([0.02, 0.01]), "dt": 1e-3,
                "nsteps": rng.randint(1, 10), "precision": rng.choice(["f64acc", "kahan"])}
    if kind == "hermite":
        n = _size(rng, 512, 131072)
        return {"kind": kind, "n": n, "masses": masses, "eps": eps, "dt": 1e-4,
                "nsteps": max(1, min(rng.randint(1, 5), int(4e10 / (float(n) * n)))),
                "precision": rng.choice(["f64acc", "kahan"])}
    if kind == "adjoint":
        n = _size(rng, 512, 32768)
        nsteps = max(4, min(rng.randint(4, 20), int(1e10 / (float(n) * n))))
        return {"kind": kind, "n": n, "masses": masses, "eps": rng.choice([0.02, 0.01, 5e-3]),
                "dt": 1e-3, "nsteps": nsteps, "segment": rng.choice([4, 10]),
                "mode": rng.choice(["reverse", "recompute"]),
                "precision": rng.choice(["f64acc", "kahan"])}
    if kind == "labels":
        return {"kind": kind, "n": _size(rng, 512, 131072), "masses": masses,
                "eps": rng.choice([0.02, 0.01]), "precision": "fp32"}
    return {"kind": kind, "n": _size(rng, 256, 40000), "masses": masses, "eps": eps,
            "precision": "fp64"}


def _cluster_sizes(case):
    """The batch's cluster sizes: log-uniform, the same for every seed."""
    return ics.batched_sizes(case["b"], 1, case["nmin"], case["nmax"])


def _particles(case, seed):
    if case["kind"] == "batched":
        return ics.batched_plummer(case["b"], seed, sizes=_cluster_sizes(case))
    if case["masses"] == "lognormal":
        return ics.plummer_lognormal(case["n"], seed)
    return ics.plummer(case["n"], seed)


def _gpu(x):
    return torch.as_tensor(x, dtype=torch.float64).to(DEV)


def _adjoint_inputs(case, seed):
    """float32 parameters (x0, v0, log m) and the FP64 target, from the seed alone."""
    s = _particles(case, seed)
    x0, v0 = (torch.tensor(a, dtype=torch.float32) for a in (s.pos, s.vel))
    logm = torch.tensor(np.log(s.mass), dtype=torch.float32)
    # the target: the particles' own drift over the run, moved by N(0, 1e-3)
    t = case["dt"] * case["nsteps"]
    target = ics.perturb_positions(s.pos + t * s.vel, 1e-3, seed + 2)
    return x0.to(DEV), v0.to(DEV), logm.to(DEV), _gpu(target)


def prepare(case, seed):
    """What a program holds before the call: the device state, its workspace and options."""
    kind = case["kind"]
    if kind == "adjoint":
        x0, v0, logm, target = _adjoint_inputs(case, seed)
        return {"case": case, "target": target,
                "params": [p.requires_grad_(True) for p in (x0, v0, logm)]}
    s = _particles(case, seed)
    if kind == "step":
        stream = torch.cuda.Stream() if case["graph"] else None
        sysm = api.System(s.pos, s.vel, s.mass, case["eps"], precision=case["precision"],
                          stream=stream, use_graph=case["graph"])
        return {"case": case, "system": sysm, "stream": stream}
    if kind == "batched":
        sysm = api.System(s.pos, s.vel, s.mass, case["eps"], offsets=s.offsets,
                          precision=case["precision"])
        return {"case": case, "system": sysm}
    st = {"case": case, "pos": _gpu(s.pos), "vel": _gpu(s.vel), "mass": _gpu(s.mass)}
    st["opts"] = binding.make_opts(case["precision"])
    st["ws"] = binding.workspace(case["n"], 1, st["opts"])
    if kind == "hermite":
        st["acc"] = torch.empty_like(st["pos"])
        st["jerk"] = torch.empty_like(st["pos"])
        st["valid"] = False
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind in ("step", "batched"):
        s = st["system"]
        s.step(case["dt"], case["nsteps"])
        if kind == "step" and case["energy"]:
            return s.pos, s.vel, s.energy()
        return s.pos, s.vel
    if kind == "hermite":
        binding.nb_hermite4(st["pos"], st["vel"], st["mass"], case["eps"], st["acc"], st["jerk"],
                            st["valid"], case["dt"], case["nsteps"], st["ws"], st["opts"])
        st["valid"] = True  # a(x), j(x) of the last evaluation serve the next call
        return st["pos"], st["vel"]
    if kind == "adjoint":
        x0, v0, logm = st["params"]
        xT, _ = adjoint.simulate(x0.double(), v0.double(), logm.double().exp(), case["eps"],
                                 case["dt"], case["nsteps"], segment=case["segment"],
                                 precision=case["precision"], mode=case["mode"])
        loss = (((xT - st["target"]) ** 2).sum() / case["n"]).float()
        return loss.detach(), *torch.autograd.grad(loss, st["params"])
    acc, pot = api.forces(st["pos"], st["mass"], case["eps"], precision=case["precision"],
                          ws=st["ws"])
    return (acc.float(), pot.float()) if kind == "labels" else (acc, pot)


def work(case):
    """FP32 (FP64 for FP64 pairs) operations over each unordered pair once, and each
    particle's inputs and outputs once.

    A pair's acceleration and potential on both particles: displacement 3, r^2 6,
    r^-1 1, r^-3 2, the two weights 2, six multiply-adds 12, two for the potential
    where it is asked for 4.  With the jerk: relative velocity 3, d.w 5, its factor 3,
    the jerk vector 6, six more multiply-adds 12.  The VJP of a pair: displacement,
    r^2 and powers 13, the weighted difference of the cotangents 9, three dot products
    15, the gradient vector 10, both particles' sums 12; its forces are counted apart.
    """
    kind = case["kind"]
    if kind == "batched":
        z = _cluster_sizes(case).astype(float)
        n, pairs = z.sum(), 0.5 * (z * (z - 1)).sum()
        return {"bytes": n * (48 + 8) + n * 48, "flops": 26 * pairs * case["nsteps"]}
    n = float(case["n"])
    pairs = 0.5 * n * (n - 1)
    if kind == "step":
        return {"bytes": n * (72 + 8) + n * 72, "flops": 26 * pairs * case["nsteps"]}
    if kind == "hermite":
        return {"bytes": n * (96 + 8) + n * 96, "flops": 55 * pairs * case["nsteps"]}
    if kind == "adjoint":
        # forward evaluations, one VJP a position and the positions' recovery
        k = case["nsteps"]
        return {"bytes": n * (28 + 24) + n * 28,
                "flops": pairs * (26 * (k + 1) + 59 * (k + 1) + 26 * k)}
    return {"bytes": n * 32 + n * (16 if kind == "labels" else 32), "flops": 30 * pairs}


# ------------------------------------------------------------------ 64 bits
_CHUNK = 1 << 24  # pairs at a time


def _rows(n):
    step = max(1, min(n, _CHUNK // n))
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _pairs64(x, i, j, eps):
    """Displacements x_j - x_i [3][rows][n], 1 / s and its square, self pairs removed."""
    d = [x[:, c][None, :] - x[i:j, c][:, None] for c in range(3)]
    r = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps).rsqrt_()
    k = torch.arange(i, j, device=x.device)
    r[k - i, k] = 0.0
    return d, r, r * r


def _forces64(x, m, eps):
    a, p = torch.empty_like(x), torch.empty_like(m)
    for i, j in _rows(x.shape[0]):
        d, r, r2 = _pairs64(x, i, j, eps)
        p[i:j] = -(r @ m)
        t = r * r2
        for c in range(3):
            a[i:j, c] = (t * d[c]) @ m
    return a, p


def _jerk64(x, v, m, eps):
    a, jk = torch.empty_like(x), torch.empty_like(x)
    for i, j in _rows(x.shape[0]):
        d, r, r2 = _pairs64(x, i, j, eps)
        t = r * r2
        w = [v[:, c][None, :] - v[i:j, c][:, None] for c in range(3)]
        q = (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]) * r2 * -3.0
        for c in range(3):
            a[i:j, c] = (t * d[c]) @ m
            jk[i:j, c] = (t * (w[c] + q * d[c])) @ m
    return a, jk


def _vjp64(x, m, eps, cot):
    """(pos_bar, mass_bar) of sum_i cot_i . a_i(x, m)."""
    xb, mb = torch.empty_like(x), torch.empty_like(m)
    for i, j in _rows(x.shape[0]):
        d, r, r2 = _pairs64(x, i, j, eps)
        t = r * r2
        # w = m_k c_j - m_j c_k with k the row
        w = [m[i:j, None] * cot[:, c][None, :] - m[None, :] * cot[i:j, c][:, None]
             for c in range(3)]
        q = (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]) * (t * r2) * -3.0
        mb[i:j] = 0.0
        for c in range(3):
            xb[i:j, c] = (t * w[c] + q * d[c]).sum(1)
            mb[i:j] -= (t * d[c]) @ cot[:, c]
    return xb, mb


def _energy64(v, m, p):
    k = 0.5 * (m * (v * v).sum(1)).sum()
    w = 0.5 * (m * p).sum()
    return torch.stack([k, w, k + w])


def _leapfrog64(x, v, m, eps, dt, nsteps, keep=None):
    x, v = x.clone(), v.clone()
    a, p = _forces64(x, m, eps)
    for _ in range(nsteps):
        if keep is not None:
            keep.append(x.clone())
        v += 0.5 * dt * a
        x += dt * v
        a, p = _forces64(x, m, eps)
        v += 0.5 * dt * a
    return x, v, p


def exact(case, seed):
    """run(prepare(case, seed)) in 64-bit torch; None where that takes too long."""
    kind = case["kind"]
    if kind == "batched":
        s = _particles(case, seed)
        pos, vel, mass = _gpu(s.pos), _gpu(s.vel), _gpu(s.mass)
        o = s.offsets.tolist()
        if sum((b - a) ** 2 for a, b in zip(o, o[1:])) * (case["nsteps"] + 1.0) > 8e10:
            return None
        for a, b in zip(o, o[1:]):
            pos[a:b], vel[a:b], _ = _leapfrog64(pos[a:b], vel[a:b], mass[a:b], case["eps"],
                                                case["dt"], case["nsteps"])
        return pos, vel
    n = float(case["n"])
    if n * n * (case.get("nsteps", 0) + 1) > 6e10:
        return None
    if kind == "adjoint":
        p32 = _adjoint_inputs(case, seed)
        x0, v0, logm = (p.double() for p in p32[:3])
        m, target, dt, eps = logm.exp(), p32[3], case["dt"], case["eps"]
        xs = []
        x, _, _ = _leapfrog64(x0, v0, m, eps, dt, case["nsteps"], xs)
        xs.append(x)
        r = x - target
        xb, vb, mb = 2.0 * r / case["n"], torch.zeros_like(r), torch.zeros_like(m)
        for k in range(case["nsteps"], -1, -1):
            if k < case["nsteps"]:
                vb = vb + dt * xb  # the drift's adjoint, then the kicks' at x_k
            half = k in (0, case["nsteps"])
            gx, gm = _vjp64(xs[k], m, eps, (0.5 * dt if half else dt) * vb)
            xb, mb = xb + gx, mb + gm
        return (r * r).sum() / case["n"], xb, vb, mb * m
    s = _particles(case, seed)
    x, v, m = _gpu(s.pos), _gpu(s.vel), _gpu(s.mass)
    if kind == "step":
        x, v, p = _leapfrog64(x, v, m, case["eps"], case["dt"], case["nsteps"])
        return (x, v, _energy64(v, m, p)) if case["energy"] else (x, v)
    if kind == "hermite":
        h = case["dt"]
        a, j = _jerk64(x, v, m, case["eps"])
        for _ in range(case["nsteps"]):
            xp = x + v * h + a * (h * h / 2) + j * (h * h * h / 6)
            vp = v + a * h + j * (h * h / 2)
            a1, j1 = _jerk64(xp, vp, m, case["eps"])
            v1 = v + (a + a1) * (h / 2) + (j - j1) * (h * h / 12)
            x = x + (v + v1) * (h / 2) + (a - a1) * (h * h / 12)
            v, a, j = v1, a1, j1
        return x, v
    return _forces64(x, m, case["eps"])
