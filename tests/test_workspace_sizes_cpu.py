"""Workspace sizes (CPU: host arithmetic only)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def size():
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    from paper_2605_02744_gb300 import binding as B

    def f(n, **kw):
        o = B.nb_opts()
        B.lib().nb_opts_default(ctypes.byref(o))
        for k, v in kw.items():
            setattr(o, k, v)
        return B.nb_workspace_bytes(n, 1, o)

    return f


@pytest.mark.parametrize("prec", ["NB_PREC_KAHAN", "NB_PREC_FP64"])
def test_four_limb_totals_end_at_their_headroom(size, prec):
    """One accumulator takes 2^19 adds, one per block of 64 slots and a few per
    warp: above 2^24 particles the four-limb paths are not provisioned (asked for
    symmetric pairs, FP64 goes direct there)."""
    from paper_2605_02744_gb300 import binding as B
    kw = dict(precision=getattr(B, prec), pairs=B.NB_PAIRS_SYMMETRIC)
    n = 1 << 24
    assert size(n + 2048, **kw) < size(n, **kw)


@pytest.mark.parametrize("n,mb", [(1024, 34.0), (16384, 57.0), (24576, 58.0), (65536, 64.0),
                                  (1 << 20, 364.0), (1 << 24, 6000.0)])
def test_totals_share_the_other_paths_scratch(size, n, mb):
    """The 224 B a particle of the four-limb totals come out of what the FP64
    cotangents, the sort and the records need anyway, as far as that goes."""
    assert size(n) <= mb * 1e6
