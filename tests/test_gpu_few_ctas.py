"""Solves on a team of few CTAs, as on a GPU (or a slice of one) with fewer
SMs: a deletion's rotations from the kept inverse are then more than 32 a
CTA.  Bar: the parity bar (identical passive set and counters, ||x - x_oracle||
<= 1e-10 ||x_oracle||), with every test of the inverse passed."""
import pytest
import torch

from oracle import oracle as O
from paper_2108_05345_gb300 import workloads as WL
from gpu_util import assert_parity, solve

pytestmark = pytest.mark.gpu


# passive sets of about 280: one, two and five strips of 32 rotations a CTA
@pytest.mark.parametrize("ctas,k_max", [(8, 9), (8, 1), (5, 24), (2, 9), (151, 9)])
def test_removals(ctas, k_max):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm as L
    build.build()
    A, b, _ = WL.overdetermined_uniform(11, m=700, n=420)
    ref = O.nnls(A, b, k_max=k_max, trace=True)
    ctx = L.Context(700, 420)
    ctx.set_ctas(ctas)
    x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
    assert_parity(x, P, info, ref, trace=ctx.trace())
    assert not ctx.state("ctl", 16)[11:13].any()
    ctx.set_ctas(0)
    x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
    assert_parity(x, P, info, ref, trace=ctx.trace())
    for bad in (-1, 1, 100000):
        assert L.lib().lhdm_debug_set_ctas(ctx.h, bad) == L.LHDM_ERR_INVALID_ARG
    ctx.close()
