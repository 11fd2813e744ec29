"""The kept inverse of R (whole-GPU solve): the sizes where it starts (more
than 128 positions in an inner step; from the first column for blocks of at
most three), long runs of removals that rotate it, blocks on either side of a
multiple of eight columns, ill-conditioned factors, and the residual test
handing the solve to substitution.  Bar: the parity bar (identical
passive set and counters, ||x - x_oracle|| <= 1e-10 ||x_oracle||); for the
ill-conditioned factors the residual and the optimality conditions, which do
not carry the condition number."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2108_05345_gb300 import workloads as WL
from gpu_util import assert_parity, kkt, solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm
    build.build()
    return lhdm


# passive sets from below 128 to about 330 positions, with removals
@pytest.mark.parametrize("m,n,k_max", [(400, 170, 24), (420, 185, 3), (500, 260, 40), (700, 420, 9), (700, 400, 1), (333, 320, 64)])
def test_removals(L, m, n, k_max):
    A, b, _ = WL.overdetermined_uniform(11, m=m, n=n)
    ref = O.nnls(A, b, k_max=k_max, trace=True)
    ctx = L.Context(m, n)
    x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
    assert_parity(x, P, info, ref, trace=ctx.trace())
    ctx.close()


@pytest.mark.parametrize("k_max", [1, 16])
@pytest.mark.parametrize("kappa", [1e5, 1e10, 1e13])
def test_ill_conditioned(L, k_max, kappa):
    A, b, _ = WL.conditioned_overdetermined(5, m=600, n=300, kappa=kappa)
    ref = O.nnls(A, b, k_max=k_max)
    ctx = L.Context(600, 300)
    x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
    assert info["status"] == ref["status"] == 0
    assert abs(info["resid_norm"] - ref["resid_norm"]) <= 1e-9 * ref["resid_norm"]
    # w on the support is zero up to the residual's rounding: 600 products,
    # each within eps ||a|| ||b||
    lo, wz, wp = kkt(A, b, x, info["tol_w"])
    assert lo >= 0.0 and wz <= 2 * info["tol_w"]
    assert wp <= 600 * 2.3e-16 * np.linalg.norm(A, axis=0).max() * (np.linalg.norm(b) + np.linalg.norm(A[:, P] * x[P], axis=0).sum())
    ctx.close()


def test_given_up(L):
    # the tests forced to fail in inner steps: with one column a block the
    # inverse is there at the first deletion, whose rotations are tested (the
    # chain takes over); with 24 an inner step makes it and tests the residual
    # of its solve (substitution takes over)
    A, b, _ = WL.overdetermined_uniform(11, m=500, n=260)
    ctx = L.Context(500, 260)
    ctx.force_commit_guard(1)
    for k_max, word in ((1, 12), (24, 11)):
        ref = O.nnls(A, b, k_max=k_max, trace=True)
        x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
        assert ctx.state("ctl", 16)[word] > 0  # the test failed, so the inverse was in use until then
        assert_parity(x, P, info, ref, trace=ctx.trace())
    ctx.close()


def test_nearly_dependent_columns(L):
    # thirty columns paired with copies that differ by 1e-8, all of them in the
    # solution (tol_w = 1e-15): cond about 1.5e9; the error an FP64 solve may
    # have is n eps cond ||x||
    rng = np.random.default_rng(3)
    m, n0, d = 500, 150, 30
    A = rng.uniform(size=(m, n0))
    A = np.asfortranarray(np.hstack([A, A[:, :d] + 1e-8 * rng.normal(size=(m, d))]))
    x0 = rng.uniform(0.1, 1, size=n0 + d)
    b = A @ x0
    ctx = L.Context(m, n0 + d)
    x, P, _, info = solve(L, ctx, A, b, k_max=1, tol_w=1e-15, max_outer=400)
    assert info["status"] == 0 and len(P) == n0 + d
    assert info["resid_norm"] <= 1e-11
    assert np.linalg.norm(x - x0) <= (n0 + d) * 2.3e-16 * 1.5e9 * np.linalg.norm(x0)
    ctx.close()
