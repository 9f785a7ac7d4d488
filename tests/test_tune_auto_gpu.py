"""tune="auto" keeps the library's own kernel where that is the fastest."""
import pytest
import torch

from paper_2605_02744_gb300 import api, binding, ics, tune as T

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cache(tmp_path, monkeypatch):
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    binding.lib()
    monkeypatch.setenv("NB_TUNE_CACHE", str(tmp_path / "t.json"))


@pytest.mark.parametrize("n", [1024, 16384])
def test_auto_is_not_a_direct_shape(n):
    """The row kernel and the warp-granular one take half the direct shapes' time
    or less at these sizes."""
    s = ics.plummer(n, seed=1)
    pos, mass = torch.tensor(s.pos, device="cuda"), torch.tensor(s.mass, device="cuda")
    a, p = api.forces(pos, mass, 0.01, tune="auto")
    assert T.lookup("force", "f64acc", n) == {}
    b, q = api.forces(pos, mass, 0.01)
    assert torch.equal(a, b) and torch.equal(p, q)
    g = api.System(s.pos, s.vel, s.mass, 0.01, tune="auto")
    assert g.opts.tune.contents.threads == 0


def test_direct_pairs_still_get_a_shape():
    s = ics.plummer(2000, seed=1)
    pos, mass = torch.tensor(s.pos, device="cuda"), torch.tensor(s.mass, device="cuda")
    api.forces(pos, mass, 0.01, tune="auto", pairs="direct")
    best = T.lookup("force-direct", "f64acc", 2000)
    assert best["threads"] > 0 and T.lookup("force", "f64acc", 2000) is None


def test_entries_made_without_the_untuned_kernel_are_not_read():
    name = T._key("force", "f64acc", 1024)
    assert "force+" in name
    T._store(name.replace("force+", "force"), {"tune": {"threads": 128}, "ms": 1.0})
    assert T.lookup("force", "f64acc", 1024) is None
