"""The first append of a solve that keeps the inverse of R goes from the
inverse's extension to the commit without a team barrier; with more than
135168 columns the commit's first words in shared memory reach the
extension's last ones, so the extension has to end with a CTA barrier.
Checked in the source; on the GPU such a solve must match the oracle with
every test of the inverse passed."""
import os
import re

import pytest
import torch

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_05345_gb300", "csrc")


def test_extension_ends_with_a_barrier():
    with open(os.path.join(CSRC, "lhdm_solve.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    i = text.index("{", text.index("void inv_extend("))
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
        if depth == 0:
            break
    assert text[i:j - 1].rstrip().endswith("__syncthreads();")


@pytest.mark.gpu
@pytest.mark.parametrize("k_max", [1, 3])
def test_many_columns(k_max):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle as O
    from paper_2108_05345_gb300 import build, lhdm as L, workloads as WL
    from gpu_util import assert_parity, solve
    build.build()
    A, b, _ = WL.gaussian_recovery(60, 140000, 4, 5, unit_columns=True)
    ref = O.nnls(A, b, k_max=k_max, trace=True)
    ctx = L.Context(*A.shape)
    x, P, _, info = solve(L, ctx, A, b, k_max=k_max)
    assert_parity(x, P, info, ref, trace=ctx.trace())
    assert not ctx.state("ctl", 16)[11:13].any()
    ctx.close()
