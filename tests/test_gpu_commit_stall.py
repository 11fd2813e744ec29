"""A tensor-core commit whose waits run out leaves nothing in flight: the last
arrivals its matrix products wait for are left out, so the issuing warp, the
warps that wait for free slots and the ones that wait for the products all
give up (after 4 s), with bulk copies and earlier products under way.  The
solve reports the timeout and the next one on the same context matches the
oracle.  Sixteen and more than 48 reflectors: one and four operand tiles."""
import pytest
import torch

from oracle import oracle as O
from paper_2108_05345_gb300 import workloads as WL
from gpu_util import assert_parity, dev, solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,s,k_max", [(300, 1600, 60, 16), (1200, 1700, 300, 64)])
def test_commit_gives_up_and_recovers(m, n, s, k_max):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm as L
    build.build()
    A, b, _ = WL.gaussian_recovery(m, n, s, 3, unit_columns=True)
    ref = O.nnls(A, b, k_max=k_max, trace=True)
    ctx = L.Context(m, n)
    At, bt = dev(L, A, b)
    ctx.inject(L.LHDM_INJECT_COMMIT_STALL)
    _, _, info = ctx.solve(At, bt, L.default_params(k_max=k_max))
    assert info["status"] == L.LHDM_ERR_TIMEOUT
    ctx.inject(0)
    for _ in range(2):
        x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
        assert_parity(x, P, info, ref, trace=ctx.trace())
    ctx.close()


def test_refused_bits():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import lhdm as L
    ctx = L.Context(8, 8)
    assert L.lib().lhdm_debug_inject(ctx.h, 1 << 20) == L.LHDM_ERR_INVALID_ARG
    assert L.lib().lhdm_debug_inject(None, 0) == L.LHDM_ERR_INVALID_ARG
    ctx.close()
