"""One workspace for problems of several sizes, options and entry points: every
result is bitwise the one of a fresh workspace, whatever the calls before left
behind."""
import numpy as np
import pytest
import torch

from paper_2605_02744_gb300 import binding, ics
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu

EPS = 0.01
SHAPE = dict(threads=512, i_per_thread=2, tile_j=1024, stages=2, ctas_per_sm=1)
FORCES = [dict(precision="f64acc"), dict(precision="fp32"), dict(precision="fp64"),
          dict(precision="kahan", pairs="symmetric", positions="split"),
          dict(precision="f64acc", pairs="direct"), dict(precision="kahan", tune=SHAPE),
          dict(precision="f64acc", positions="adaptive")]
NMAX = 66000


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    binding.lib()


class Calls:
    """Every entry point on one system; run(ws) gives the outputs by name."""

    def __init__(self, n):
        s = ics.plummer_lognormal(n, seed=n)
        self.n = n
        self.pos, self.vel, self.mass = dev(s.pos), dev(s.vel), dev(s.mass)
        self.cot = dev(np.random.default_rng(n).normal(size=(n, 3)))

    def _pair(self, rows=None):
        n = self.n if rows is None else rows
        return (torch.empty((n, 3), dtype=torch.float64, device="cuda"),
                torch.empty(n, dtype=torch.float64, device="cuda"))

    def names(self):
        some = [str(i) for i in range(len(FORCES))]
        if self.n > 30000:
            some = ["0", "1", "4"]
        return (["forces" + i for i in some] + ["vjp", "vjp-direct", "jerk", "range", "step"] +
                (["step-fp64"] if self.n < 30000 else []))

    def opts(self, name):
        if name.startswith("forces"):
            return binding.make_opts(**FORCES[int(name[6:])])
        if name == "vjp-direct":
            return binding.make_opts("f64acc", pairs="direct")
        return binding.make_opts("fp64" if name == "step-fp64" else "kahan")

    def run(self, name, ws):
        o, n = self.opts(name), self.n
        if name.startswith("forces"):
            out = self._pair()
            binding.nb_forces(self.pos, self.mass, EPS, *out, ws, o)
        elif name.startswith("vjp"):
            out = self._pair()
            binding.nb_forces_vjp(self.pos, self.mass, EPS, self.cot, None, *out, ws, o)
        elif name == "jerk":
            out = (torch.empty_like(self.pos), torch.empty_like(self.pos))
            binding.nb_forces_jerk(self.pos, self.vel, self.mass, EPS, *out, None, ws, o)
        elif name == "range":
            out = self._pair(n - n // 3)
            binding.nb_forces_range(self.pos, self.mass, n // 3, n, EPS, *out, ws, o)
        else:
            x, v = self.pos.clone(), self.vel.clone()
            acc, pot = self._pair()
            st = binding.make_state(x, v, self.mass, acc, pot, EPS, ws)
            binding.nb_step(st, 1e-4, 2, o)
            e = torch.empty(3, dtype=torch.float64, device="cuda")
            binding.nb_energy(st, e, o)
            out = (x, v, acc, pot, e)
        assert binding.nb_poll_status(ws, o) == binding.NB_OK
        return out


def fresh(calls, name):
    return calls.run(name, binding.workspace(calls.n, 1, calls.opts(name)))


def shared_workspace():
    sizes = [binding.nb_workspace_bytes(NMAX, 1, binding.make_opts(**kw)) for kw in FORCES]
    return torch.zeros(max(sizes), dtype=torch.uint8, device="cuda")


def test_sizes_down_and_up_on_one_workspace():
    ws = shared_workspace()
    sizes = [20001, 10000, 2047, 300, 4097, 60, NMAX, 1000, 20001, NMAX]
    calls = {n: Calls(n) for n in set(sizes)}
    want = {(n, k): fresh(c, k) for n, c in calls.items() for k in c.names()}
    bad = []
    for n in sizes:
        for k in calls[n].names():
            got = calls[n].run(k, ws)
            if not all(torch.equal(a, b) for a, b in zip(got, want[n, k])):
                bad.append((n, k))
    assert not bad, bad


@pytest.mark.parametrize("n", [60, 300, 4097, 9000, 30000, NMAX])
def test_only_the_status_block_is_kept(n):
    """Beyond its first 256 bytes a workspace may hold anything."""
    calls = Calls(n)
    ws = shared_workspace()
    for k in calls.names():
        ws[256:] = 0x5a
        assert all(torch.equal(a, b) for a, b in zip(calls.run(k, ws), fresh(calls, k))), k


def test_graph_replay_after_another_size():
    """A captured step loop of the warp-granular path replays on a workspace that
    another size used in between."""
    n, other = 6000, Calls(9000)
    s = ics.plummer(n, seed=1)
    st = torch.cuda.Stream()
    out = []
    for graph in (False, True):
        o = binding.make_opts("f64acc", stream=st, use_graph=graph)
        x, v, m = dev(s.pos), dev(s.vel), dev(s.mass)
        acc, pot = torch.zeros_like(x), torch.zeros_like(m)
        ws = shared_workspace()
        state = binding.make_state(x, v, m, acc, pot, EPS, ws)
        torch.cuda.synchronize()
        for _ in range(3):  # acc_valid = 0, then one graph replayed
            binding.nb_step(state, 1e-4, 3, o)
            torch.cuda.synchronize()
            other.run("vjp", ws)
            torch.cuda.synchronize()
        out.append((x, v, acc, pot))
    assert all(torch.equal(a, b) for a, b in zip(*out))
