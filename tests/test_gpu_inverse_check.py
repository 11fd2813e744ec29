"""What a solve with the kept inverse of R returns is tested itself: the
residual of the corrected y, row by row, against the rounding of a solve; the
residual before the correction says nothing certain about it.  A host
example of the difference; the returned y of ill-conditioned solves with
long runs of removals; and each place where the test is read (beside the
commit, beside the x update, at the end of the inner loop) made to fail:
substitution takes over and the decisions and counters stay the oracle's."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2108_05345_gb300 import workloads as WL
from gpu_util import assert_parity, solve

U = 2.0 ** -53


def within_rounding(R, y, rhs, slack=0.0):
    """Rows of R y = rhs within (16 + 8 min(k, 32)) u of their largest term or
    of their sum (slack: more of u times the row's absolute sum)."""
    k = len(y) - np.arange(len(y))
    t = np.triu(R) * y[None, :]
    s = np.abs(t.sum(1))
    scale = np.maximum(s, np.abs(t).max(1))
    d = np.abs(rhs - t.sum(1))
    return d <= (16 + 8 * np.minimum(k, 32)) * U * scale + slack * U * np.abs(t).sum(1)


def test_small_residual_before_the_correction_is_no_guarantee():
    # E = I - R X takes 2^-27 of row 2 into row 1 and 2^-10 of row 1 into row 0;
    # row 1's right-hand side is small because its terms cancel.  One product
    # leaves 2^-27 of every row's largest term, the second one 2^-37 of row 0's.
    R = np.array([[1.0, 0.0, 0.0], [0.0, 1.0, -1.0], [0.0, 0.0, 1.0]])
    E = np.zeros((3, 3))
    E[0, 1], E[1, 2] = 2.0 ** -10, 2.0 ** -27
    X = np.linalg.inv(R) @ (np.eye(3) - E)
    rhs = np.array([1.0, 2.0 ** -17, 1.0])
    y = X @ rhs
    d = rhs - R @ y
    assert (np.abs(d) <= 2.0 ** -26 * np.abs(R * y[None, :]).max(1)).all()  # the rule lets it through
    y = y + X @ d
    assert np.abs(rhs - R @ y)[0] > 2.0 ** -38
    assert within_rounding(R, y, rhs).tolist() == [False, True, True]  # the test does not
    y = y + X @ (rhs - R @ y)
    assert within_rounding(R, y, rhs).all()


def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm
    build.build()
    return lhdm


@pytest.mark.gpu
@pytest.mark.parametrize("kappa,k_max", [(1e6, 1), (1e8, 1), (1e10, 1), (1e13, 1), (1e6, 16), (1e10, 16)])
def test_returned_solution_is_within_rounding(kappa, k_max):
    L = lib()
    A, b, _ = WL.conditioned_overdetermined(6, m=1000, n=500, kappa=kappa)
    ctx = L.Context(1000, 500)
    x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
    assert info["status"] == 0 and info["n_inner"] > 100
    # rhs and y_P are the last solve's: an inner step's, or the last append's
    # over the positions before it
    last = ctx.trace()[-1]
    nP = info["n_passive"]
    n0 = nP if last[2] else nP - int(last[1])
    sl = ctx.state("rslot", 500)
    R = ctx.state("R", 500 * 500).reshape(500, 500)[sl[:n0], :n0].T.astype(np.longdouble)
    y, rhs = ctx.state("yP", 500)[:n0], ctx.state("rhs", 500)[:n0]
    assert within_rounding(R, y.astype(np.longdouble), rhs, slack=16).all()
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("where,m,n,seed,k_max", [("append", 600, 300, 11, 1), ("append", 500, 260, 11, 24),
                                                  ("inner", 600, 400, 11, 32), ("inner", 420, 300, 13, 40),
                                                  ("inner", 700, 420, 11, 64), ("inner", 600, 300, 11, 1)])
def test_refused_solution(where, m, n, seed, k_max):
    L = lib()
    A, b, _ = WL.overdetermined_uniform(seed, m=m, n=n)
    ref = O.nnls(A, b, k_max=k_max, trace=True)
    ctx = L.Context(m, n)
    ctx.inject(L.LHDM_INJECT_CHECK_APPEND if where == "append" else L.LHDM_INJECT_CHECK_INNER)
    for _ in range(2):
        x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
        assert_parity(x, P, info, ref, trace=ctx.trace())
        assert ctx.state("ctl", 16)[11] > 0
    ctx.inject(0)
    x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
    assert_parity(x, P, info, ref, trace=ctx.trace())
    assert ctx.state("ctl", 16)[11] == 0
    ctx.close()


@pytest.mark.gpu
def test_refused_solution_with_signs():
    L = lib()
    A, b = WL.signed_overdetermined(3, m=500, n=250)[:2]
    for mode in (1, 2):
        ref = O.nnls_signed(A, b, sign_flip=mode == 2, k_max=24)
        ctx = L.Context(500, 250)
        for inject in (0, L.LHDM_INJECT_CHECK_APPEND | L.LHDM_INJECT_CHECK_INNER):
            ctx.inject(inject)
            x, P, _, info = solve(L, ctx, A, b, k_max=24, mode=mode)
            assert P.tolist() == ref["passive"].tolist()
            assert np.linalg.norm(x - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])
            assert (info["n_outer"], info["n_inner"]) == (ref["n_outer"], ref["n_inner"])
        ctx.close()
