"""The forms of the block-reflector commit at the edges of their ranges,
against the oracle: tensor cores with 16 to 64 reflectors (one to four
operand tiles), 8 and 16 columns a batch, rows over one exact accumulation
(1024) and ragged; the FP64 forms for few columns per CTA (the whole GPU on
a narrow problem) and for many (one CTA per instance), with V in shared
memory whole and in parts.  Bar: identical passive set and counters,
||x - x_oracle|| <= 1e-10 ||x_oracle|| (the parity bar of every GPU test)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2108_05345_gb300 import workloads as WL
from gpu_util import assert_parity, dev, solve

pytestmark = pytest.mark.gpu

# m, n, nonzeros, k_max
CASES = [(300, 1600, 60, 16), (300, 1600, 60, 32), (263, 1601, 55, 20), (1200, 1000, 150, 64), (1200, 1700, 300, 64),
         (2100, 1300, 180, 32), (300, 400, 40, 7), (90, 700, 12, 9)]


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm
    build.build()
    return lhdm


def instance(case):
    m, n, s, k = case
    A, b, _ = WL.gaussian_recovery(m, n, s, 3, unit_columns=True)
    return A, b, k


@pytest.mark.parametrize("case", CASES)
def test_whole_gpu(L, case):
    A, b, k = instance(case)
    ref = O.nnls(A, b, k_max=k, trace=True)
    ctx = L.Context(*A.shape)
    for guard in (0, 1):  # 1: tensor cores wherever they can run, then handed to FP64
        ctx.force_commit_guard(guard)
        x, P, _, info = solve(L, ctx, A, b, k_max=k)
        assert_parity(x, P, info, ref, trace=ctx.trace())
    ctx.close()


def test_one_cta_per_instance(L):
    refs, As, bs = [], [], []
    for case in CASES + [(150, 300, 20, 32), (420, 500, 60, 48)]:
        if case[1] > 1700:
            continue
        A, b, k = instance(case)
        refs.append(O.nnls(A, b, k_max=24, trace=True))
        At, bt = dev(L, A, b)
        As.append(At)
        bs.append(bt)
    B = L.Batch(As, bs, L.default_params(k_max=24))
    B.run()
    torch.cuda.synchronize()
    for x, p, info, ref in zip(B.xs, B.ps, B.info(), refs):
        ps = p.cpu().numpy()
        assert_parity(x.cpu().numpy(), ps[ps >= 0], info, ref)
    B.close()


@pytest.mark.parametrize("mode", [0, 1])
def test_one_cta_many_removals(L, mode):
    # noise: blocks of every size, removals, passive sets up to the row count
    As, bs, refs = [], [], []
    for i, m in enumerate((72, 121, 200, 333)):
        A, b, _ = WL.batched_instance(40 + i, m)
        k = (8, 40)[mode]
        refs.append(O.nnls(A, b, k_max=k, trace=True))
        At, bt = dev(L, A, b)
        As.append(At)
        bs.append(bt)
    B = L.Batch(As, bs, L.default_params(k_max=(8, 40)[mode]))
    B.run()
    torch.cuda.synchronize()
    for x, p, info, ref in zip(B.xs, B.ps, B.info(), refs):
        ps = p.cpu().numpy()
        assert_parity(x.cpu().numpy(), ps[ps >= 0], info, ref)
    B.close()
