"""One CTA per instance with blocks of 33 to 64 reflectors (three and four
operand tiles of the tensor-core commit) and each instance's own k_max.  Bar:
identical passive set and counters, ||x - x_oracle|| <= 1e-10 ||x_oracle||."""
import pytest
import torch

from oracle import oracle as O
from paper_2108_05345_gb300 import workloads as WL
from gpu_util import assert_parity, dev

pytestmark = pytest.mark.gpu

# m, n, nonzeros
CASES = [(1000, 400, 200), (1200, 1000, 150), (1500, 1300, 260)]


@pytest.mark.parametrize("k", [33, 40, 48, 64])
def test_blocks(k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm as L
    build.build()
    refs, As, bs = [], [], []
    for m, n, s in CASES:
        A, b, _ = WL.gaussian_recovery(m, n, s, 3, unit_columns=True)
        refs.append(O.nnls(A, b, k_max=k, trace=True))
        At, bt = dev(L, A, b)
        As.append(At)
        bs.append(bt)
    # the blocks in question occur
    assert any(max(int(t[1]) for t in r["trace"]) > 32 for r in refs)
    B = L.Batch(As, bs, L.default_params(k_max=k))
    B.run()
    torch.cuda.synchronize()
    for x, p, info, ref in zip(B.xs, B.ps, B.info(), refs):
        ps = p.cpu().numpy()
        assert_parity(x.cpu().numpy(), ps[ps >= 0], info, ref)
    B.close()
