"""Results do not depend on what device or shared memory held before: NaN is
written over freed device memory (and with it through the SMs' L1, whose
lines are the shared memory of the next launch) right before a context is made
and a solve runs.  The sizes end a triangular solve in a short 64-position
block (passive sets passing 129 .. 191) and cover one CTA, the batch and the
signed mode.  Bar: the parity bar, and the same bits with a second fill."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2108_05345_gb300 import workloads as WL
from gpu_util import assert_parity, solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm
    build.build()
    return lhdm


def leave(value):
    ts = [torch.full((1 << k,), value, dtype=torch.float64, device="cuda") for k in (19, 20, 21, 22, 23, 24, 26)]
    torch.cuda.synchronize()
    del ts
    torch.cuda.empty_cache()


def scaled(m, n):
    A, b, _ = WL.overdetermined_uniform(5, m=m, n=n)
    rng = np.random.default_rng(16)
    rs, cs = 2.0 ** rng.integers(-15, 16, size=m), 2.0 ** rng.integers(-2, 3, size=n)
    return np.asfortranarray(A * rs[:, None] * cs[None, :]), b * rs


@pytest.mark.parametrize("m,n,k_max,mode", [(700, 350, 32, 0), (700, 350, 12, 0), (420, 260, 1, 0), (130, 70, 24, 0), (300, 160, 16, 1)])
def test_single(L, m, n, k_max, mode):
    A, b = scaled(m, n)
    out = []
    for value in (float("nan"), 1e300):
        leave(value)
        ctx = L.Context(m, n)
        x, P, _, info = solve(L, ctx, A, b, k_max=k_max, mode=mode)
        if mode == 0:
            assert_parity(x, P, info, O.nnls(A, b, k_max=k_max, trace=True), trace=ctx.trace())
        assert info["status"] == 0 and np.isfinite(x).all()
        out.append(x)
        ctx.close()
    assert np.array_equal(out[0], out[1])


def test_batch(L):
    probs = [scaled(m, n) for m, n in ((700, 350), (300, 150), (65, 64), (420, 260))]
    out = []
    for value in (float("nan"), 1e300):
        leave(value)
        dev = [(L.colmajor(torch.from_numpy(np.ascontiguousarray(A)).cuda()), torch.from_numpy(b).cuda()) for A, b in probs]
        batch = L.Batch([d[0] for d in dev], [d[1] for d in dev], L.default_params(k_max=16))
        leave(value)
        batch.run()
        torch.cuda.synchronize()
        out.append([x.cpu().numpy() for x in batch.xs])
        batch.close()
    for (A, b), x0, x1 in zip(probs, *out):
        ref = O.nnls(A, b, k_max=16)
        assert np.linalg.norm(x0 - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])
        assert np.array_equal(x0, x1)
