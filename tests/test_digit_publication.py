"""The panel's reflector digits are written to global memory by ordinary
stores and read by bulk copies (the async proxy), in the whole-GPU solve by
other CTAs: each side needs an unrestricted proxy fence beside the barrier
between them.  The order is checked in the source (a digit buffer that is
one panel old gives wrong numbers only when the timing allows it); on the
GPU, solves whose digit buffers hold another problem's digits must repeat
bit for bit."""
import os
import re

import numpy as np
import pytest
import torch

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_05345_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body(text, head):
    """The braced body of the function whose definition contains head."""
    i = text.index("{", text.index(head))
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
        if depth == 0:
            return text[i:j]


def test_both_sides_fence_the_proxies():
    eng, sol = source("lhdm_engine.cuh"), source("lhdm_solve.cuh")
    assert '"fence.proxy.async;"' in body(eng, "void fence_proxy_async_all()")
    publish = body(sol, "void publish_digits()")
    assert "fence_proxy_async_all()" in publish and "__threadfence()" in publish
    for panel in ("bool panel(const int* s_J)", "bool panel_rows("):
        b = body(sol, panel)
        last = max(b.rindex("vd_store_row("), b.rindex("vd_store_tail("))
        assert "publish_digits()" in b[last:], panel
    commit = body(sol, "int commit_tc(")
    first = commit.index("bulk_g2s(")
    assert "fence_proxy_async_all();" in commit[:first]
    # the fence is every thread's, and a CTA barrier passes it on to the copying thread
    assert "__syncthreads()" in commit[commit.index("fence_proxy_async_all();"):first]


@pytest.mark.gpu
def test_repeats_bit_for_bit():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm as L, workloads as WL
    from gpu_util import dev
    build.build()
    probs = [dev(L, *WL.gaussian_recovery(m, n, s, 7, unit_columns=True)[:2])
             for m, n, s in ((300, 1600, 60), (260, 1200, 50))]
    ctx = L.Context(300, 1600)
    for k in (16, 24, 64):
        prm = L.default_params(k_max=k)
        first = [ctx.solve(A, b, prm)[0].cpu().numpy().copy() for A, b in probs]
        for _ in range(6):
            for (A, b), x in zip(probs, first):
                assert np.array_equal(ctx.solve(A, b, prm)[0].cpu().numpy(), x)
        batch = L.Batch([A for A, _ in probs] * 8, [b for _, b in probs] * 8, prm)
        for _ in range(3):
            batch.run()
            torch.cuda.synchronize()
            xs = [x.cpu().numpy().copy() for x in batch.xs]
            for i, x in enumerate(xs):
                assert np.array_equal(x, xs[i & 1])
        batch.close()
    ctx.close()
