"""Device memory of a context: W, R and, for the first 3072 positions of every
slot, R's inverse (kept only up to there), beside panel scratch that grows
with m + n alone."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(6000, 6000), (8192, 5000), (2000, 3000)])
def test_bytes(m, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm as L
    build.build()
    L.Context(64, 64).close()  # the library's kernels are loaded
    cap = min(m, n)
    before = torch.cuda.mem_get_info()[0]
    ctx = L.Context(m, n)
    used = before - torch.cuda.mem_get_info()[0]
    ctx.close()
    # 400 doubles a row: 64 reflectors, their digits (8 x 64 bf16), the
    # triangular solve's 64-blocks, vectors; 24 MB for what does not grow
    bound = 8 * (m * n + cap * cap + cap * min(cap, 3072) + 400 * (m + n)) + (24 << 20)
    assert 8 * (m * n + cap * cap) < used <= bound, (used, bound)


@pytest.mark.parametrize("nz", [2940, 3000])
def test_more_positions_than_the_inverse_has(nz):
    """Past 3072 passive columns, with an inner step that goes from 3075 back
    to 3070: slots past 3072 hold rows of the inverse then.  The solution is the
    least-squares one on its columns, and optimal."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_05345_gb300 import build, lhdm as L
    build.build()
    m, n = 3400, 3300
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    A = torch.rand((n, m), generator=g, device="cuda", dtype=torch.float64).t()
    x0 = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) + 0.2
    x0[nz:] = 0.0
    b = A @ x0 + 0.3 * torch.randn(m, generator=g, device="cuda", dtype=torch.float64)
    ctx = L.Context(m, n)
    x, p, info = ctx.solve(A, b, L.default_params(k_max=64))
    ctx.close()
    assert info["status"] == L.LHDM_OK and info["n_passive"] > 3072
    P = p[p >= 0].long()
    z = torch.linalg.lstsq(A[:, P], b[:, None]).solution[:, 0]
    w = A.t() @ (b - A @ x)
    scale = float(A.norm(dim=0).max() * b.norm())
    out = torch.ones(n, dtype=torch.bool, device="cuda")
    out[P] = False
    assert float((x[P] - z).norm()) <= 1e-9 * float(z.norm())
    assert bool((x >= 0).all()) and float(x[out].abs().sum()) == 0.0
    assert float(w[out].max()) <= 1e-10 * scale and float(w[P].abs().max()) <= 1e-10 * scale
