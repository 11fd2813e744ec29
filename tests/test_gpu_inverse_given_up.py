"""A solve that fails its residual test gives the kept inverse of R up for the
deletions that follow too, not for solves alone.  The test of the solves is
made to fail by itself (the deletions' own test stays as it is); the count of
deletions that took their rotations from the inverse shows who was asked.
Bar: the parity bar of the other tests."""
import pytest
import torch

from oracle import oracle as O
from paper_2108_05345_gb300 import workloads as WL
from gpu_util import assert_parity, solve

pytestmark = pytest.mark.gpu


# the first inner step with more than 128 positions, whose solve makes the
# inverse, is followed by one to three more in the same outer step
@pytest.mark.parametrize("m,n,seed,k_max", [(600, 400, 11, 32), (700, 420, 13, 32), (420, 300, 13, 40)])
def test_deletions_follow_the_solves(m, n, seed, k_max):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm as L
    build.build()
    A, b, _ = WL.overdetermined_uniform(seed, m=m, n=n)
    ref = O.nnls(A, b, k_max=k_max, trace=True)
    ctx = L.Context(m, n)
    for inject in (0, L.LHDM_INJECT_SOLVE_TEST):
        ctx.inject(inject)
        x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
        assert_parity(x, P, info, ref, trace=ctx.trace())
        ctl = ctx.state("ctl", 16)
        assert (ctl[11] > 0) == (inject != 0)
        assert (ctl[13] > 0) == (inject == 0), ctl
    ctx.close()
