"""The FP64 commit of columns that do not fit shared memory whole: more rows
than the tensor-core form takes (16384), and blocks of four reflectors at
9000 rows, with 1 to 16 columns per CTA (whole GPU) and one CTA for all.
Bar: identical passive set and counters, ||x - x_oracle|| <= 1e-10
||x_oracle|| (the parity bar of every GPU test).

Its time follows the columns a CTA has: the commit phase keeps a tenth of the
1.26 TFLOP/s the GPU has in FP64 (measured 0.3 and 0.65 TFLOP/s with 2 and 7
columns per CTA; on 32 lanes whatever the columns it was 0.03 and 0.11)."""
import pytest
import torch

from oracle import oracle as O
from paper_2108_05345_gb300 import workloads as WL
from gpu_util import assert_parity, dev, solve

pytestmark = pytest.mark.gpu

# m, n, nonzeros, k_max
CASES = [(17000, 120, 12, 8), (17000, 400, 20, 16), (16900, 1000, 30, 32), (17000, 1400, 40, 40), (17500, 2300, 30, 32),
         (9000, 900, 20, 4)]
# the same kernel takes the small ones of a mixed batch
ONE_CTA = [(17000, 40, 10, 8), (600, 300, 40, 8), (16500, 33, 12, 12), (9000, 50, 10, 4), (700, 400, 30, 4), (90, 60, 9, 4)]


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm
    build.build()
    return lhdm


def instance(case):
    m, n, s, k = case
    A, b, _ = WL.gaussian_recovery(m, n, s, 5, unit_columns=True)
    return A, b, k


@pytest.mark.parametrize("case", CASES)
def test_whole_gpu(L, case):
    A, b, k = instance(case)
    ref = O.nnls(A, b, k_max=k, trace=True)
    ctx = L.Context(*A.shape)
    x, P, _, info = solve(L, ctx, A, b, k_max=k)
    assert_parity(x, P, info, ref, trace=ctx.trace())
    ctx.close()


def test_one_cta_per_instance(L):
    for k in sorted({c[3] for c in ONE_CTA}):
        refs, As, bs = [], [], []
        for case in (c for c in ONE_CTA if c[3] == k):
            A, b, _ = instance(case)
            refs.append(O.nnls(A, b, k_max=k, trace=True))
            At, bt = dev(L, A, b)
            As.append(At)
            bs.append(bt)
        B = L.Batch(As, bs, L.default_params(k_max=k))
        B.run()
        torch.cuda.synchronize()
        for x, p, info, ref in zip(B.xs, B.ps, B.info(), refs):
            ps = p.cpu().numpy()
            assert_parity(x.cpu().numpy(), ps[ps >= 0], info, ref)
        B.close()


@pytest.mark.parametrize("n,k", [(300, 8), (1000, 32)])
def test_commit_rate(L, n, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    m = 20000
    A = torch.rand((n, m), generator=g, device="cuda", dtype=torch.float64).t()
    x = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (torch.arange(n, device="cuda") % 2)
    b = A @ x + 1e-2 * torch.randn(m, generator=g, device="cuda", dtype=torch.float64)
    ctx = L.Context(m, n)
    best = 0.0
    for _ in range(2):
        ctx.solve(A, b, L.default_params(k_max=k))
        ms, flops = ctx.profile()
        best = max(best, flops["commit"] / ms["commit"] * 1e-9)
    ctx.close()
    assert best > 0.126, "commit at %.3f TFLOP/s" % best
