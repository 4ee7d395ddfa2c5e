"""What the performance of this framework is measured on: one pass each through its public entry points.

The kinds of pass are those a regression run is made of: the packed build, the dual objective (value and gradient), the
contraction on its own, the dual Hessian-vector product, the full Hessian, and a whole solve with its primal weights.  Sizes
are those of the seeded workloads of ``synth`` (plain FP64 n = 40, full FP32 n = 400, order 6 n = 80, Nystrom BF16 n' = 600,
lambda path n' = 300 with 512 problems, Dexter-shaped d = 20,000), those of the thesis's other runs, and odd
ones between them.

Storage is a case's own: "f64", "f32" or "bf16".  Passes over FP32 or BF16 storage accumulate in FP32; the entry points hand
some of their results out in FP64 containers, which a program of that precision keeps in FP32, and so does ``run``.
"""
import math

import torch

import paper_2003_10482_gb300 as tk

LAMBDA = 1.0 / 0.86  # gamma = 0.86, the value of the thesis's synthetic runs
BYTES = {"f64": 8, "f32": 4, "bf16": 2}


def listed():
    return [
        # the smallest call: one objective evaluation of the plain FP64 workload, as every solver step repeats it
        {"name": "objective_f64_n40", "kind": "objective", "m": 4, "n": 40, "d": 10, "storage": "f64", "B": 1},
        # the headline: one objective evaluation of the full FP32 workload
        {"name": "objective_f32_n400", "kind": "objective", "m": 4, "n": 400, "d": 100, "storage": "f32", "B": 1},
        # the higher-order workload's contraction: many small triangles
        {"name": "contract_f32_m6_n80", "kind": "contract", "m": 6, "n": 80, "d": 50, "storage": "f32", "B": 1},
        # a conjugate-gradient step of Newton-CG, at an odd size
        {"name": "hvp_f32_n351", "kind": "hvp", "m": 4, "n": 351, "d": 100, "storage": "f32", "B": 1},
        # a conjugate-gradient step of the mixed BF16 / FP32 Nystrom solve: the largest tensor
        {"name": "hvp_bf16_n600", "kind": "hvp", "m": 4, "n": 600, "d": 200, "storage": "bf16", "B": 1},
        # the build of the full FP32 workload
        {"name": "build_f32_n400_d100", "kind": "build", "m": 4, "n": 400, "d": 100, "storage": "f32", "feat": "linear"},
        # the Dexter-shaped build: few points, very many sparse features
        {"name": "build_f32_n200_d20000", "kind": "build", "m": 4, "n": 200, "d": 20000, "storage": "f32", "feat": "linear"},
        # the thesis's Wpbc-shaped build in its own precision
        {"name": "build_f64_n120_d32", "kind": "build", "m": 4, "n": 120, "d": 32, "storage": "f64", "feat": "linear"},
        # the Newton matrix of one problem of the lambda path
        {"name": "hessian_f32_n300", "kind": "hessian", "m": 4, "n": 300, "d": 80, "storage": "f32"},
        # all 512 problems of the lambda path x folds in one objective and gradient pass
        {"name": "contract_f32_n300_B512", "kind": "contract", "m": 4, "n": 300, "d": 80, "storage": "f32", "B": 512},
        # one conjugate-gradient step of 64 problems of the path together
        {"name": "hvp_f32_n300_B64", "kind": "hvp", "m": 4, "n": 300, "d": 80, "storage": "f32", "B": 64},
        # a whole call at the size of the thesis's synthetic runs (more features than points): 8 lambdas solved by
        # full-Hessian Newton, and their primal weights
        {"name": "solve_f32_n250_d2000_B8", "kind": "solve", "m": 4, "n": 250, "d": 2000, "storage": "f32", "B": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["objective", "contract", "hvp", "build", "build", "hessian", "batch", "solve"])
    storage = rng.choice(["f32", "f32", "bf16", "f64"])
    if kind == "build":
        m = rng.choice([3, 4, 4, 6])
        n = _log(rng, *{3: (40, 800), 4: (30, 400), 6: (12, 40)}[m])
        N = math.comb(n + m - 1, m)
        # at most half of the Dexter-shaped build's multiply-adds (FP64 units are some 70 times slower)
        most = (1.5e12 if storage != "f64" else 2e11) / (2.0 * N)
        d = _log(rng, 8, max(8, min(20000, int(most))))
        return {"kind": "build", "m": m, "n": n, "d": d, "storage": storage, "feat": rng.choice(["linear", "linear", "poly", "exp"])}
    if kind == "hessian":
        m = rng.choice([3, 4, 4])
        n = _log(rng, 40, {3: 400, 4: 300}[m])
        return {"kind": "hessian", "m": m, "n": n, "d": _log(rng, 8, 100), "storage": storage}
    if kind == "batch":  # several problems in one pass: contraction or Hessian-vector product
        storage = rng.choice(["f32", "bf16"])
        if rng.random() < 0.5:
            return {"kind": "contract", "m": rng.choice([3, 4]), "n": _log(rng, 64, 300), "d": _log(rng, 8, 80), "storage": storage, "B": _log(rng, 40, 512)}
        return {"kind": "hvp", "m": rng.choice([3, 4]), "n": _log(rng, 40, 300), "d": _log(rng, 8, 80), "storage": storage, "B": _log(rng, 2, 64)}
    if kind == "solve":
        storage = rng.choice(["f32", "f64"])
        n = _log(rng, 30, 240 if storage == "f32" else 80)
        return {"kind": "solve", "m": 4, "n": n, "d": _log(rng, n, 2000), "storage": storage, "B": _log(rng, 1, 8)}
    m = rng.choice([3, 4, 4, 6])
    n = _log(rng, *{3: (40, 1000), 4: (30, 400), 6: (12, 80)}[m])
    return {"kind": kind, "m": m, "n": n, "d": _log(rng, 8, 100), "storage": storage, "B": 1}


# ------------------------------------------------------------------ inputs
def _inputs(case, seed):
    """X (n x d FP64), and what the pass needs beside it: dual vectors, a direction, labels, lambdas."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")

    m, n, d, B = case["m"], case["n"], case["d"], case.get("B", 1)
    X = normal(n, d)
    if d >= 5000:  # many features: sparse rows, as in text data
        X = torch.where(torch.rand(n, d, generator=g, dtype=torch.float64, device="cuda") < 0.005, X, torch.zeros_like(X))
    if case.get("feat", "linear") != "linear":  # arguments of the nonlinear maps of order one
        X = X * float(d) ** (-1.0 / m)
    w = torch.zeros(d, dtype=torch.float64, device="cuda")
    s = min(10, d)
    w[:s] = torch.sign(normal(s)) * (1.0 - 0.3 * torch.rand(s, generator=g, dtype=torch.float64, device="cuda"))
    y = X @ w + 0.05 * normal(n)
    A = normal(B, n) / math.sqrt(n)
    V = normal(B, n)
    lam = torch.logspace(-0.3, 0.3, B, dtype=torch.float64, device="cuda") if case["kind"] == "solve" else torch.tensor([LAMBDA], dtype=torch.float64, device="cuda")
    if B == 1 and case["kind"] != "contract":
        A, V = A[0], V[0]
    if case["kind"] == "contract" and case["storage"] != "f64":
        A = A.float()
    return X, A, V, y, lam


def prepare(case, seed):
    X, A, V, y, lam = _inputs(case, seed)
    state = {"case": case, "X": X, "A": A, "V": V, "y": y, "lam": lam}
    if case["kind"] != "build":
        state["K"] = tk.tk_build_packed(X, case["m"], storage=case["storage"])
    return state


def _kept(state, *tensors):
    """Results in the precision of the pass."""
    dtype = torch.float64 if state["case"]["storage"] == "f64" else torch.float32
    return [t.to(dtype) for t in tensors]


def run(state):
    case = state["case"]
    kind, m, n = case["kind"], case["m"], case["n"]
    if kind == "build":
        return tk.tk_build_packed(state["X"], m, storage=case["storage"], feat=case["feat"], degree=2 if case["feat"] == "poly" else 1)
    K = state["K"]
    if kind == "objective":
        return _kept(state, *tk.tk_objective(K, m, n, state["A"], state["y"], state["lam"]))
    if kind == "contract":
        return _kept(state, *tk.tk_contract(K, m, n, state["A"]))
    if kind == "hvp":
        return _kept(state, tk.tk_dual_hvp(K, m, n, state["A"], state["V"], state["lam"]))
    if kind == "hessian":
        return _kept(state, tk.tk_hessian(K, m, n, state["A"]))
    tol = dict(tol=1e-10) if case["storage"] == "f64" else dict(tol=0.0, rel_gap=1e-9, max_iter=30)
    A, _, _ = tk.tk_solve_dual(K, m, n, state["y"], state["lam"], method="newton_full", **tol)
    return _kept(state, A, tk.tk_primal(state["X"], A, m))


def work(case):
    m, n, d, B, es = case["m"], case["n"], case["d"], case.get("B", 1), BYTES[case["storage"]]
    N = math.comb(n + m - 1, m)
    if case["kind"] == "build":  # the feature products and their sums
        return {"bytes": N * es + 8 * n * d, "flops": 2 * N * d}
    if case["kind"] == "hessian":  # per entry: its own place, and a product with a on either side
        return {"bytes": N * es + 8 * n * n + 8 * n, "flops": 6 * N}
    if case["kind"] == "solve":  # some six Newton steps of all problems: a pass over the tensor and a Cholesky factor each
        return {"bytes": 6 * N * es + 8 * B * n, "flops": 6 * B * (6 * N + n**3 // 3)}
    per = 6 if case["kind"] == "hvp" else 4
    return {"bytes": N * es + 24 * B * n, "flops": per * N * B}


# ------------------------------------------------------------------ the same in 64 bits
def _packed(X, m, feat, storage):
    """Sum over features of the products of every sorted m-tuple of rows, in the packed order, by blocks of the leading indices."""
    n, d = X.shape
    out = torch.empty(math.comb(n + m - 1, m), dtype=torch.float64, device=X.device)
    lead = [()]
    for _ in range(m - 3):
        lead = [p + (i,) for p in lead for i in range(p[-1] if p else 0, n)]
    at, rows = 0, max(1, min(16, (1 << 26) // (n * d)))
    index = torch.arange(n, device=X.device)
    for p in lead:
        w = torch.ones(d, dtype=torch.float64, device=X.device)
        for i in p:
            w = w * X[i]
        for i0 in range(p[-1] if p else 0, n, rows):
            i1 = min(i0 + rows, n)
            Y = (X[i0:i1] * w)[:, None, :] * X[None, i0:, :]
            T = (Y.reshape(-1, d) @ X[i0:].T).reshape(i1 - i0, n - i0, n - i0)
            c = index[i0:]
            keep = (c[None, :, None] >= index[i0:i1, None, None]) & (c[None, None, :] >= c[None, :, None])
            v = T[keep]
            out[at : at + v.numel()] = v
            at += v.numel()
    if feat == "poly":
        out = out * out
    elif feat == "exp":
        out = torch.exp(out)
    return out


def _newton(X, y, lam, m):
    """The minimiser of sum((X^T a)^m)/m + lam/2 |a|^2 - <y, a>."""
    def value(a):
        return ((X.T @ a) ** m).sum() / m + 0.5 * lam * (a @ a) - y @ a

    a = torch.zeros_like(y)
    for _ in range(100):
        u = X.T @ a
        grad = X @ u ** (m - 1) + lam * a - y
        H = (m - 1) * (X * u ** (m - 2)) @ X.T + lam * torch.eye(len(y), dtype=y.dtype, device=y.device)
        p = -torch.linalg.solve(H, grad)
        t, f, slope = 1.0, value(a), float(grad @ p)
        while t > 1e-3 and float(value(a + t * p) - f) > 1e-4 * t * slope + 1e-13 * abs(float(f)):
            t *= 0.5
        a = a + t * p
        if float(p.norm()) <= 1e-14 * float(a.norm()):
            break
    return a


def exact(case, seed):
    kind, m, n = case["kind"], case["m"], case["n"]
    X, A, V, y, lam = _inputs(case, seed)
    if kind == "build":
        # the tensor is made block by block of its first m - 2 indices: too many small ones above order 4
        if math.comb(n + m - 4, max(m - 3, 0)) * (n // 16 + 1) > 60000:
            return None
        return _packed(X, m, case["feat"], case["storage"])
    # the linear tensor kernel is sum_k (X_k)^(x m): its contractions have closed forms in u = X^T a
    A, V = A.double(), V.double()
    U = A @ X
    if kind == "objective":
        grad = U ** (m - 1) @ X.T + lam * A - y
        F = (U**m).sum(-1) / m + 0.5 * lam * (A * A).sum(-1) - A @ y
        return [F.reshape(-1), grad, grad.norm(dim=-1).reshape(-1)]
    if kind == "contract":
        return [U ** (m - 1) @ X.T, (U**m).sum(-1).reshape(-1)]
    if kind == "hvp":
        return [(m - 1) * (U ** (m - 2) * (V @ X)) @ X.T + lam * V]
    if kind == "hessian":
        return [(X * U ** (m - 2)) @ X.T]
    A = torch.stack([_newton(X, y, float(v), m) for v in lam])
    u = A @ X
    return [A, torch.sign(u) * u.abs() ** (m - 1)]
