"""Below the range of the adaptive symmetric path one workspace size serves a
system under every precision and pairs option (CPU: sizes only)."""
import pytest


@pytest.mark.parametrize("n", [64, 1000, 4800, 16384, 24575])
def test_one_size_below_the_adaptive_range(n):
    import paper_2605_02744_gb300 as pkg
    pkg.build()
    from paper_2605_02744_gb300 import binding as B
    import ctypes

    def size(**kw):
        o = B.nb_opts()
        B.lib().nb_opts_default(ctypes.byref(o))
        for k, v in kw.items():
            setattr(o, k, v)
        return B.nb_workspace_bytes(n, 1, o)

    base = size()
    for prec in (B.NB_PREC_FP32, B.NB_PREC_KAHAN, B.NB_PREC_FP64):
        for pairs in (B.NB_PAIRS_DEFAULT, B.NB_PAIRS_DIRECT):
            assert size(precision=prec, pairs=pairs) == base
    assert size(test_unissued_stage=2) == base and size(positions=B.NB_POS_ADAPTIVE) == base
