"""The NNLS work that users of this package have it do, as cases to be timed.

A case is one call (or one training step) through the package's public entry
points: single solves on device or host buffers, the allocation-free solve,
the l1 sweep, the positivity trick, batches of uneven instances and the
differentiable layer.  Sizes, block sizes and value distributions are those
of the package's workloads, tests and benchmark; `draw` gives more of the
same ranges.  Inputs are made on the GPU from a seed (column-major float64,
as the entry points take them).
"""
import math

import torch

from paper_2108_05345_gb300 import layer as nnls_layer
from paper_2108_05345_gb300 import lhdm

DEV = "cuda"
F8 = torch.float64


def listed():
    return [
        # a fixed-memory real-time loop: the smallest problem, by the entry
        # point that allocates nothing; launch and barrier latency is all of it
        {"name": "static_65x64", "kind": "static", "m": 65, "n": 64, "k_max": 4},
        # one small fit inside a model: the layer on a single ragged problem,
        # forward and backward
        {"name": "layer_single_257x131", "kind": "layer1", "m": 257, "n": 131, "k_max": 16},
        # the paper's small sparse recovery: a few blocked steps, no removals
        {"name": "recovery_256x512", "kind": "recovery", "m": 256, "n": 512, "s": 25, "k_max": 8},
        # a mid-size dense fit whose data lives on the host (copies included)
        {"name": "host_1000x500", "kind": "host", "m": 1000, "n": 500, "k_max": 32},
        # a regularisation sweep: l1-NNLS for three weights
        {"name": "l1_sweep_512x1024", "kind": "l1", "m": 512, "n": 1024, "s": 40, "k_max": 32},
        # wide sparse recovery (2048 x 8192): many columns, few steps
        {"name": "recovery_2048x8192", "kind": "recovery", "m": 2048, "n": 8192, "s": 128, "k_max": 64},
        # unconstrained-sign least squares by the positivity trick with sign flips
        {"name": "signed_flip_2048x1024", "kind": "signed", "m": 2048, "n": 1024, "mode": 2, "k_max": 32},
        # the classical one-column method on a mid-size dense fit
        {"name": "lh_2048x1024", "kind": "dense", "m": 2048, "n": 1024, "k_max": 1},
        # ill-conditioned dense fit: the solve with the most removals
        {"name": "conditioned_2048x1024", "kind": "conditioned", "m": 2048, "n": 1024, "kappa": 1e6, "k_max": 32},
        # the headline: one large dense overdetermined fit
        {"name": "dense_4096x2048", "kind": "dense", "m": 4096, "n": 2048, "k_max": 32},
        # a training step of the layer on a batch: forward and backward
        {"name": "layer_batch_64x512x1024", "kind": "layer", "count": 64, "m": 512, "n": 1024, "s": 40, "k_max": 32},
        # many uneven instances in one launch, block size by the built-in rule
        {"name": "batch_1024_uneven", "kind": "batch", "count": 1024, "m_lo": 64, "m_hi": 512, "sizes": 0, "k_max": 0},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, even over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["static", "layer1", "recovery", "host", "l1", "signed", "dense", "dense", "lh", "conditioned",
                       "layer", "batch"])
    k = rng.choice([4, 8, 16, 32, 64])
    if kind == "static":
        m = _log(rng, 24, 256)
        if m >= 128 and rng.random() < 0.4:  # wide: sparse recovery
            return {"kind": kind, "m": m, "n": int(m * rng.uniform(1.2, 2.0)), "s": max(8, m // 16), "k_max": k}
        return {"kind": kind, "m": m, "n": max(8, int(m * rng.uniform(0.4, 1.0))), "k_max": k}
    if kind == "layer1":
        m = _log(rng, 48, 1024)
        return {"kind": kind, "m": m, "n": max(16, int(m * rng.uniform(0.3, 0.8))), "k_max": k}
    if kind == "recovery":
        m = _log(rng, 256, 2048)
        return {"kind": kind, "m": m, "n": int(m * rng.uniform(2.0, 4.0)), "s": max(8, int(m * rng.uniform(0.03, 0.09))),
                "k_max": max(8, k)}
    if kind == "l1":
        m = _log(rng, 128, 1024)
        return {"kind": kind, "m": m, "n": int(m * rng.uniform(1.5, 2.5)), "s": max(4, m // 13), "k_max": max(8, k)}
    if kind == "signed":
        m = _log(rng, 256, 2048)
        return {"kind": kind, "m": m, "n": max(64, int(m * rng.uniform(0.25, 0.5))), "mode": rng.choice([1, 2]), "k_max": max(8, k)}
    if kind in ("dense", "host"):
        m = _log(rng, 128, 4096)
        return {"kind": kind, "m": m, "n": max(32, int(m * rng.uniform(0.25, 0.5))), "k_max": max(8, k)}
    if kind == "lh":
        m = _log(rng, 128, 2048)
        return {"kind": "dense", "m": m, "n": max(32, int(m * rng.uniform(0.25, 0.5))), "k_max": 1}
    if kind == "conditioned":
        m = _log(rng, 256, 2048)
        return {"kind": kind, "m": m, "n": m // 2 - rng.randrange(0, 40), "kappa": rng.choice([1e5, 1e6]), "k_max": max(8, k)}
    if kind == "layer":
        m = _log(rng, 64, 512)
        return {"kind": kind, "count": _log(rng, 4, 96), "m": m, "n": 2 * m - rng.randrange(0, 9), "s": max(4, m // 13), "k_max": rng.choice([8, 16, 32])}
    lo = _log(rng, 32, 200)
    return {"kind": "batch", "count": _log(rng, 16, 700), "m_lo": lo, "m_hi": rng.randrange(lo, 480) + 20,
            "sizes": rng.randrange(1000), "k_max": rng.choice([0, 0, 8, 32])}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=F8)


def _uniform(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=F8)


def _cols(At):
    """(n, m) rows = columns of A -> the column-major (m, n) matrix."""
    return At.t()


def _spread(g, n, s):
    """n values, s of them at random places uniform on (0.1, 1], the rest 0."""
    x = torch.zeros(n, device=DEV, dtype=F8)
    x[torch.randperm(n, generator=g, device=DEV)[:s]] = 1.0 - 0.9 * _uniform(g, s)
    return x


def _conditioned(g, m, n, kappa):
    """U diag(sigma) V^T, sigma log-spaced over 1 .. 1/kappa, unit columns."""
    r = min(m, n)
    U = torch.linalg.qr(_normal(g, m, r))[0]
    V = torch.linalg.qr(_normal(g, n, r))[0]
    sigma = torch.logspace(0.0, -math.log10(kappa), r, device=DEV, dtype=F8)
    A = (U * sigma) @ V.t()
    A /= torch.linalg.vector_norm(A, dim=0, keepdim=True)
    return lhdm.colmajor(A)


def _inputs(case, seed):
    """A (column-major) and b of a single-problem case."""
    g, kind, m, n = _gen(seed), case["kind"], case["m"], case["n"]
    if "s" in case and kind != "l1":  # sparse nonnegative x, unit columns, noiseless
        A = _cols(_normal(g, n, m))
        A /= torch.linalg.vector_norm(A, dim=0, keepdim=True)
        b = A @ _spread(g, n, case["s"])
    elif kind in ("static", "layer1", "host", "dense", "conditioned"):
        # half of x zero, the rest uniform; a noisy right-hand side
        A = _conditioned(g, m, n, case["kappa"]) if kind == "conditioned" else _cols(_uniform(g, n, m))
        x = (1.0 - _uniform(g, n)) * (torch.randperm(n, generator=g, device=DEV) < n - n // 2)
        b = A @ x + 1e-2 * _normal(g, m)
    elif kind == "signed":
        A = _cols(_normal(g, n, m) / math.sqrt(m))
        b = A @ _normal(g, n) + _normal(g, m)
    else:  # l1: signed sparse x, noise
        A = _cols(_normal(g, n, m) / math.sqrt(m))
        sign = torch.where(_uniform(g, n) < 0.5, -1.0, 1.0).to(F8)
        b = A @ (_spread(g, n, case["s"]) * sign) + 1e-3 * _normal(g, m)
    return A, b


L1_WEIGHTS = (1.0, 10.0, 100.0)


def _batch_sizes(case):
    g = torch.Generator()
    g.manual_seed(case["sizes"])
    return torch.randint(case["m_lo"], case["m_hi"] + 1, (case["count"],), generator=g).tolist()


def _batch_inputs(case, seed):
    """Uneven instances: n = 2m, A ~ N(0, 1/m), 10 % nonzeros, noise N(0, 1e-3)."""
    g, ms = _gen(seed), _batch_sizes(case)
    flat = _normal(g, sum(2 * m * m for m in ms))
    noise = math.sqrt(1e-3) * _normal(g, sum(ms))
    mag = 1.0 - 0.9 * _uniform(g, sum(2 * m for m in ms))
    order = _uniform(g, sum(2 * m for m in ms))
    As, bs, o, q = [], [], 0, 0
    for m in ms:
        n = 2 * m
        A = _cols(flat[o:o + n * m].view(n, m))
        A /= math.sqrt(m)
        x = mag[2 * q:2 * q + n] * (order[2 * q:2 * q + n].argsort().argsort() < max(1, round(0.1 * n)))
        As.append(A)
        bs.append(A @ x + noise[q:q + m])
        o += n * m
        q += m
    return As, bs


def _layer_inputs(case, seed):
    """A batch of equal problems as a model holds it, with targets for x."""
    g, c, m, n = _gen(seed), case["count"], case["m"], case["n"]
    A = _normal(g, c, m, n) / math.sqrt(m)
    x0 = torch.stack([_spread(g, n, case["s"]) for _ in range(c)])
    b = torch.einsum("cmn,cn->cm", A, x0) + math.sqrt(1e-3) * _normal(g, c, m)
    return A, b, x0 + 1e-2 * _normal(g, c, n)


def _layer1_target(case, seed):
    return _uniform(_gen(seed + 77), case["n"])


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "prm": lhdm.default_params(k_max=case["k_max"], mode=case.get("mode", 0))}
    if kind == "batch":
        st["A"], st["b"] = _batch_inputs(case, seed)
        ns = [A.shape[1] for A in st["A"]]
        # the outputs of all instances side by side, as one buffer each
        st["x"] = torch.empty(sum(ns), device=DEV, dtype=F8)
        st["p"] = torch.empty(sum(ns), device=DEV, dtype=torch.int32)
        st["xs"], st["ps"] = list(st["x"].split(ns)), list(st["p"].split(ns))
        st["infos"] = torch.zeros(case["count"] * 7, device=DEV, dtype=F8)
        st["ctx"] = lhdm.Context(max(A.shape[0] for A in st["A"]), max(ns), case["count"])
    elif kind == "layer":
        A, b, st["target"] = _layer_inputs(case, seed)
        st["A"], st["b"] = A.requires_grad_(), b.requires_grad_()
        st["layer"] = nnls_layer.NNLSLayer(case["m"], case["n"], case["count"], k_max=case["k_max"])
    elif kind == "layer1":
        A, b = _inputs(case, seed)
        st["A"], st["b"], st["target"] = A.requires_grad_(), b.requires_grad_(), _layer1_target(case, seed)
        st["layer"] = nnls_layer.NNLSLayer(case["m"], case["n"], k_max=case["k_max"])
    elif kind == "host":
        A, b = _inputs(case, seed)
        host = torch.empty(case["n"], case["m"], dtype=F8, pin_memory=True)
        host.copy_(A.t())
        st["A"], st["b"] = host.numpy().T, b.cpu().pin_memory().numpy()
        st["ctx"] = lhdm.Context(case["m"], case["n"])
    else:
        st["A"], st["b"] = _inputs(case, seed)
        if kind == "l1":
            st["ctx"] = lhdm.Context(case["m"] + 1, 2 * case["n"])
        elif kind != "static":
            st["ctx"] = lhdm.Context(case["m"], case["n"])
    return st


def run(st):
    kind = st["kind"]
    if kind == "static":
        _, x, p, _ = lhdm.solve_noalloc(st["A"], st["b"], st["prm"])
        return {"x": x, "passive": p}
    if kind in ("layer", "layer1"):
        x = st["layer"](st["A"], st["b"])
        loss = 0.5 * (x - st["target"]).square().sum()
        dA, db = torch.autograd.grad(loss, (st["A"], st["b"]))
        return {"x": x.detach(), "dA": dA, "db": db}
    if kind == "batch":
        st["ctx"].solve_batched(st["A"], st["b"], st["prm"], st["xs"], st["ps"], st["infos"])
        return {"x": st["x"], "passive": st["p"]}
    if kind == "l1":
        return [{"x": x, "passive": p, "status": info["status"]} for x, p, info in st["ctx"].l1_path(st["A"], st["b"], L1_WEIGHTS, st["prm"])]
    if kind == "host":
        x, p, info = st["ctx"].solve_host(st["A"], st["b"], st["prm"])
    else:
        x, p, info = st["ctx"].solve(st["A"], st["b"], st["prm"])
    return {"x": x, "passive": p, "status": info["status"]}


# ---------------------------------------------------------------- work
def _solve_work(m, n, p, k):
    """One solve that ends with p passive columns in blocks of k: the QR of
    those columns and a dual product A^T r for every block."""
    p = min(p, m, n)
    return 8 * m * n + 8 * m + 12 * n, 2 * m * p * p - 2 * p ** 3 / 3 + 2 * m * n * math.ceil(p / max(1, k))


def work(case):
    kind, k = case["kind"], case["k_max"]
    if kind == "batch":
        ws = [_solve_work(m, 2 * m, m, k or 16) for m in _batch_sizes(case)]
        return {"bytes": sum(w[0] for w in ws), "flops": sum(w[1] for w in ws)}
    m, n = case["m"], case["n"]
    if kind in ("layer", "layer1"):
        c = case.get("count", 1)
        w = _solve_work(m, n, m if kind == "layer" else 0.7 * n, k)
        # and dA, db written
        return {"bytes": c * (w[0] + 8 * m * n + 8 * m + 8 * n), "flops": c * (w[1] + 4 * m * n)}
    if kind == "l1":
        ws = [_solve_work(m, n, p * case["s"], k) for p in (0.2, 1.0, 1.8)]
        return {"bytes": sum(w[0] for w in ws) + 2 * 12 * n, "flops": sum(w[1] for w in ws)}
    p = case.get("s") or {"signed": n, "conditioned": 0.55 * n}.get(kind, 0.7 * n)
    w = _solve_work(m, n, p, k)
    return {"bytes": w[0], "flops": w[1]}


# ---------------------------------------------------------------- 64-bit values
def _least_squares(A, b, P):
    """Least squares on the columns P by QR, refined once."""
    Q, R = torch.linalg.qr(A[:, P])
    z = torch.linalg.solve_triangular(R, (Q.t() @ b)[:, None], upper=True)[:, 0]
    r = b - A[:, P] @ z
    return z + torch.linalg.solve_triangular(R, (Q.t() @ r)[:, None], upper=True)[:, 0]


def _active_set(A, b, most=32, steps=600):
    """Plain active-set NNLS: the `most` best columns enter at a time while
    every new coefficient stays positive, else one; ends at the optimality
    conditions, which are checked on the refined solution (None if they fail).
    Used where the minimiser is unique, so the way to it does not matter."""
    m, n = A.shape
    G, c = A.t() @ A, A.t() @ b
    scale = float(A.square().sum(0).max().sqrt() * b.norm())
    x = torch.zeros(n, device=A.device, dtype=F8)
    P = torch.zeros(n, device=A.device, dtype=torch.bool)

    def solve():
        idx = P.nonzero()[:, 0]
        z = torch.zeros_like(x)
        z[idx] = _least_squares(A, b, idx) if ill else torch.cholesky_solve(c[idx][:, None], torch.linalg.cholesky(G[idx][:, idx]))[:, 0]
        return z

    ill = False
    add = most
    for _ in range(steps):
        w = (A.t() @ (b - A @ x)).masked_fill(P, -math.inf)
        top = torch.topk(w, min(add, n - int(P.sum())))
        new = top.indices[top.values > max(1e-12 * scale, 0.3 * float(top.values[0]))] if top.values.numel() else top.indices
        if new.numel() == 0:
            break
        P[new] = True
        progress = False
        while True:
            try:
                z = solve()
            except torch.linalg.LinAlgError:
                ill = True
                z = solve()
            if bool((z[P] > 0).all()):
                x, progress = z, True
                break
            bad = P & (z <= 0)
            t = float((x[bad] / (x[bad] - z[bad])).min())
            progress |= t > 0
            x = x + t * (z - x)
            out = P & ((x <= 1e-15 * x.max()) & (z <= 0))
            x[out] = 0.0
            P &= ~out
            if not bool(P.any()):
                break
        add = most if progress else 1
    idx = P.nonzero()[:, 0]
    x = torch.zeros_like(x)
    x[idx] = _least_squares(A, b, idx)
    w = (A.t() @ (b - A @ x))[~P]
    if bool((x[idx] <= 0).any()) or (w.numel() and float(w.max()) > 1e-11 * scale):
        return None
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("layer", "batch"):
        return None  # more columns than rows and noise: every solve ends at one of many minimisers
    A, b = _inputs(case, seed)
    rest = {"passive": None} if kind == "static" else {"passive": None, "status": None}
    if "s" in case and kind != "l1":
        # noiseless: the sparse vector itself
        g = _gen(seed)
        _normal(g, case["n"], case["m"])
        return {"x": _spread(g, case["n"], case["s"]), **rest}
    if kind == "signed":
        x = _least_squares(A, b, torch.arange(case["n"], device=DEV))
        return {"x": torch.cat([x.clamp_min(0), (-x).clamp_min(0)]), **rest}
    if kind == "l1":
        one, zero = torch.ones(1, 2 * case["n"], device=DEV, dtype=F8), torch.zeros(1, device=DEV, dtype=F8)
        xs = [_active_set(torch.cat([one, torch.cat([v * A, -v * A], 1)]), torch.cat([zero, v * b])) for v in L1_WEIGHTS]
        return [{"x": x, **rest} for x in xs]
    x = _active_set(A, b)
    if kind != "layer1":
        return {"x": x, **rest}
    if x is None:
        return None
    # dL/dx = x - target on the passive set P: u = (A_P^T A_P)^-1 g_P,
    # dL/db = A_P u, dL/dA_P = r u^T - (A_P u) x_P^T
    P = (x > 0).nonzero()[:, 0]
    R = torch.linalg.qr(A[:, P])[1]
    v = torch.linalg.solve_triangular(R.t(), (x - _layer1_target(case, seed))[P][:, None], upper=False)
    u = torch.linalg.solve_triangular(R, v, upper=True)[:, 0]
    db = A[:, P] @ u
    dA = torch.zeros_like(A)
    dA[:, P] = torch.outer(b - A @ x, u) - torch.outer(db, x[P])
    return {"x": x, "dA": dA, "db": db}
