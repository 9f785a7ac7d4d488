"""F64ACC adds its FP32 partial sums in FP64, on every path.

A particle at the origin, all others on one spot at distance 1: each pair term
is the partner's mass (or cotangent) itself, so the total has to be its sum
exactly.  The terms 1, 2^-25 and 2^-50 lie in different partial sums; a pair of
floats holds the first two and loses the third."""
import numpy as np
import pytest
import torch

from paper_2605_02744_gb300 import binding
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu

TERMS = (1.0, 2.0 ** -25, 2.0 ** -50)
EPS = 1e-8  # eps^2 is below half an ulp of 1 in FP32: r^-1 is 1


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    binding.lib()


def weights(n, terms, where):
    w = np.zeros(n)
    for t, i in zip(terms, where):
        w[i] = t
    return w


# N, particles that carry the terms: in three of the four warps of the row
# kernel; in three warps' ranges of one row and CTA of the symmetric kernels
CASES = [(2000, (69, 133, 197)), (5000, (200, 330, 460)), (12500, (600, 1200, 1800))]


@pytest.mark.parametrize("n,where", CASES)
@pytest.mark.parametrize("positions", ["split", "single"])
@pytest.mark.parametrize("what", ["forces", "jerk", "vjp"])
def test_total_is_the_sum_of_its_terms(n, where, positions, what):
    x = np.ones((n, 3)) * [1.0, 0.0, 0.0]
    x[0] = 0.0
    pos = dev(x)
    o = binding.make_opts("f64acc", positions=positions)
    ws = binding.workspace(n, 1, o)

    def total(terms):
        w = dev(weights(n, terms, where))
        out, other = torch.empty_like(pos), torch.empty_like(pos)
        per = torch.empty(n, dtype=torch.float64, device="cuda")
        if what == "forces":
            binding.nb_forces(pos, w, EPS, out, per, ws, o)
            assert float(-per[0]) == sum(terms)
        elif what == "jerk":
            binding.nb_forces_jerk(pos, torch.zeros_like(pos), w, EPS, out, other, per, ws, o)
            assert float(-per[0]) == sum(terms)
        else:
            cot = torch.zeros_like(pos)
            cot[:, 0] = w
            binding.nb_forces_vjp(pos, torch.ones_like(w), EPS, cot, None, out, per, ws, o)
            return -float(per[0])
        return float(out[0, 0])

    assert total(TERMS[:1]) == 1.0
    assert total(TERMS) == sum(TERMS)  # 1 + 2^-25 + 2^-50, exact in FP64
