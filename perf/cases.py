"""Performance cases of the GoDec library: what a program that uses it has it do.

Each case is one call, or one run of calls, of the public Python API
(``paper_1309_0302_gb300``) on data already on the GPU.  The inputs are the library's own
synthetic recipe: X = U V^T + S + G with Gaussian factors, gross errors on uniformly drawn
positions and Gaussian noise.  The gross errors have magnitudes well above the noise, so that
after a few iterations the support of S is the planted one and no tie of rounding decides it.

Kinds of case:
  product    one streaming product Y = Z B (``mul_ZB``) or W = Z^T C (``mul_ZtC``)
  threshold  the S-step alone on a dense residual (``hard_threshold``)
  solve      a decomposition with a context that the program keeps: from S = 0, a fixed number
             of iterations, then L (dense) and S (sorted COO)
  once       the same for a matrix that is seen once: context, iterations, results, release
  batch      many uneven problems advanced together (``GoDecBatch``), L factors kept apart
  gradient   the differentiated form's backward (``backward``) for given supports
  lingodec   LinGoDec alternations with given item features
"""
import math

import torch

import paper_1309_0302_gb300 as G


def listed():
    return [
        # one product of a small matrix: the smallest call, latency and launches
        {"name": "product_500", "kind": "product", "m": 500, "n": 500, "r": 10, "trans": False},
        # the transposed product of a ragged matrix, sizes that no tile divides
        {"name": "product_t_ragged", "kind": "product", "m": 20011, "n": 3003, "r": 21, "trans": True},
        # one product at the size of the benchmark
        {"name": "product_10000", "kind": "product", "m": 10000, "n": 10000, "r": 50, "trans": False},
        # selection of the largest 2 % of a mid-size dense residual
        {"name": "threshold_ragged", "kind": "threshold", "m": 4001, "n": 2999, "density": 0.02},
        # the paper's 500 x 500 experiment: latency-bound iterations on a cache-resident matrix
        {"name": "solve_500", "kind": "solve", "m": 500, "n": 500, "r": 10, "q": 1, "density": 0.05, "iters": 8,
         "half": False},
        # a ragged mid-size matrix that is seen once: set-up, iterations, results, release
        {"name": "once_ragged", "kind": "once", "m": 3001, "n": 2047, "r": 24, "q": 1, "density": 0.03, "iters": 6,
         "half": False},
        # the benchmark workload
        {"name": "solve_10000", "kind": "solve", "m": 10000, "n": 10000, "r": 50, "q": 2, "density": 0.01,
         "iters": 10, "half": False},
        # a video-shaped matrix (pixels x frames) at a low rank
        {"name": "solve_tall", "kind": "solve", "m": 76800, "n": 1000, "r": 3, "q": 2, "density": 0.015, "iters": 6,
         "half": False},
        # the precision form (16-bit power chain, float32 correction) on a video-shaped matrix
        {"name": "precision_tall", "kind": "solve", "m": 38400, "n": 600, "r": 6, "q": 2, "density": 0.015,
         "iters": 6, "half": True},
        # 64 uneven problems in one batch
        {"name": "batch_64", "kind": "batch", "count": 64, "lo": 256, "hi": 4096, "mix": 1309, "iters": 6},
        # gradient of unrolled q = 0 iterations with a dense loss gradient
        {"name": "gradient_4096", "kind": "gradient", "m": 4096, "n": 4096, "r": 20, "T": 4, "density": 0.02},
        # users x items with given item features
        {"name": "lingodec_items", "kind": "lingodec", "m": 20000, "n": 5000, "d": 50, "r": 10, "density": 0.01,
         "iters": 5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, lo, most):
    """Rows and columns, log-uniform from lo, with at most `most` entries."""
    while True:
        m, n = _log(rng, lo, 80000), _log(rng, lo, 12000)
        if m * n <= most:
            return m, n


def draw(rng):
    u = rng.random()
    if u < 0.3:
        m, n = _shape(rng, 300, 10 ** 8)
        return {"kind": "product", "m": m, "n": n, "r": rng.randint(1, min(64, m, n)), "trans": rng.random() < 0.5}
    if u < 0.4:
        m, n = _shape(rng, 300, 10 ** 8)
        return {"kind": "threshold", "m": m, "n": n, "density": rng.choice([0.002, 0.01, 0.02, 0.05])}
    if u < 0.75:
        m, n = _shape(rng, 300, 9 * 10 ** 7)
        half = rng.random() < 0.15
        # rank well below both dimensions, the support recoverable from the given rank
        r = rng.randint(2, max(2, min(32 if half else 50, min(m, n) // 25)))
        q = rng.choice([1, 1, 2])
        return {"kind": "solve" if rng.random() < 0.6 else "once", "m": m, "n": n, "r": r, "q": q,
                "density": rng.choice([0.005, 0.01, 0.02, 0.03]), "iters": rng.randint(6, 8),
                "half": half}
    if u < 0.83:
        return {"kind": "batch", "count": rng.randint(6, 48), "lo": 256, "hi": _log(rng, 600, 4096), "mix": rng.randint(0, 10 ** 6),
                "iters": 6}
    if u < 0.92:
        m, n = _shape(rng, 500, 16 * 10 ** 6)
        return {"kind": "gradient", "m": m, "n": n, "r": rng.randint(2, max(2, min(24, min(m, n) // 25))),
                "T": rng.randint(2, 4), "density": rng.choice([0.01, 0.02])}
    m, n = _shape(rng, 1500, 9 * 10 ** 7)
    d = rng.randint(8, 56)
    return {"kind": "lingodec", "m": m, "n": n, "d": d, "r": rng.randint(2, min(d, 16)), "density": 0.01, "iters": 5}


# ---- inputs ---------------------------------------------------------------------------------
def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _randn(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)


def _positions(g, total, density):
    """Distinct ascending positions, one drawn in each of density * total equal intervals."""
    k = max(1, int(density * total))
    width = total // k
    return torch.arange(k, device="cuda") * width + torch.randint(width, (k,), generator=g, device="cuda")


def _gross(g, count, lo=2.0, hi=10.0):
    v = lo + (hi - lo) * torch.rand(count, generator=g, device="cuda")
    return torch.where(torch.rand(count, generator=g, device="cuda") < 0.5, -v, v)


def _lowrank_sparse(g, m, n, r, density):
    X = _randn(g, m, r) @ _randn(g, n, r).T
    X += 1e-2 * _randn(g, m, n)
    pos = _positions(g, m * n, density)
    X.view(-1)[pos] += _gross(g, pos.numel())
    return X, _randn(g, n, r), pos


def _batch_shapes(case):
    g = torch.Generator().manual_seed(case["mix"])
    out = []
    for _ in range(case["count"]):
        u = torch.rand(4, generator=g, dtype=torch.float64).tolist()
        ratio = math.log(case["hi"] / case["lo"])
        m, n = (int(round(case["lo"] * math.exp(ratio * t))) for t in u[:2])
        r = 2 + int(u[2] * (min(32, min(m, n) // 25) - 1))
        out.append((m, n, r, 0.02 + 0.02 * u[3]))
    return out


def _inputs(case, seed):
    """The tensors of a case, from its seed alone."""
    kind, g = case["kind"], _gen(seed)
    if kind == "product":
        m, n, r = case["m"], case["n"], case["r"]
        Z = _lowrank_sparse(g, m, n, min(r, 16), 0.01)[0]
        return {"Z": Z, "B": _randn(g, m if case["trans"] else n, r)}
    if kind == "threshold":
        m, n = case["m"], case["n"]
        R = 1e-2 * _randn(g, m, n)
        pos = _positions(g, m * n, case["density"])
        R.view(-1)[pos] += _gross(g, pos.numel(), 0.05, 10.0)
        return {"R": R, "k": int(pos.numel())}
    if kind in ("solve", "once"):
        X, A1, pos = _lowrank_sparse(g, case["m"], case["n"], case["r"], case["density"])
        return {"X": X, "A1": A1, "k": int(pos.numel())}
    if kind == "batch":
        Xs, As, ks, rs = [], [], [], []
        for m, n, r, density in _batch_shapes(case):
            X, A1, pos = _lowrank_sparse(g, m, n, r, density)
            Xs.append(X)
            As.append(A1)
            ks.append(int(pos.numel()))
            rs.append(r)
        return {"Xs": Xs, "A1s": As, "ks": ks, "rs": rs}
    if kind == "gradient":
        m, n, r = case["m"], case["n"], case["r"]
        X, A1, pos = _lowrank_sparse(g, m, n, r, case["density"])
        sup = []
        for _ in range(case["T"] - 1):   # the planted support, part of it still moving
            keep = pos[torch.randperm(pos.numel(), generator=g, device="cuda")[:pos.numel() * 9 // 10]]
            sup.append(torch.cat([keep, _positions(g, m * n, 0.1 * case["density"])]).unique())
        gL = _randn(g, m, r) @ _randn(g, n, r).T
        return {"X": X, "A1": A1, "supports": sup, "gL": gL}
    m, n, d, r = case["m"], case["n"], case["d"], case["r"]
    F = _randn(g, n, d)
    # preferences of rank r with a weak part on every feature (the rank constraint drops it)
    W = _randn(g, m, r) @ (_randn(g, r, d) / math.sqrt(d)) + 1e-2 * _randn(g, m, d)
    X = W @ F.T
    X += 1e-2 * _randn(g, m, n)
    pos = _positions(g, m * n, case["density"])
    X.view(-1)[pos] += _gross(g, pos.numel())
    return {"X": X, "F": F, "lam": 0.5}


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "solve":
        s["ctx"] = G.GoDec(s["X"], s["A1"], case["r"], s["k"], case["q"], tol=0.0, max_iter=50,
                           precision=G.PREC_BF16_REFINE if case["half"] else G.PREC_FP32)
    elif kind == "batch":
        s["ctx"] = G.GoDecBatch(s["Xs"], s["A1s"], s["rs"], s["ks"], 1)
    elif kind == "lingodec":
        s["ctx"] = G.LinGoDec(s["X"], s["F"], case["r"], s["lam"])
    s["case"] = dict(case)
    return s


# ---- one pass -------------------------------------------------------------------------------
def _results(ctx, rel):
    idx, val = ctx.S()
    return {"L": ctx.L_dense(), "S_idx": idx, "S_val": val, "rel_err": float(rel)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "product":
        return (G.mul_ZtC if case["trans"] else G.mul_ZB)(state["Z"], state["B"])
    if kind == "threshold":
        return G.hard_threshold(state["R"], state["k"])
    if kind == "solve":
        ctx = state["ctx"]
        ctx.reset()
        return _results(ctx, ctx.iterate(case["iters"]))
    if kind == "once":
        ctx = G.GoDec(state["X"], state["A1"], case["r"], state["k"], case["q"], tol=0.0, max_iter=50,
                      precision=G.PREC_BF16_REFINE if case["half"] else G.PREC_FP32)
        try:
            return _results(ctx, ctx.iterate(case["iters"]))
        finally:
            ctx.close()
    if kind == "batch":
        batch = state["ctx"]
        batch.reset()
        batch.iterate(case["iters"])
        # L = U diag(sigma) V^T of every problem, one after the other, and their errors
        Ls, errs = [], []
        for i in range(case["count"]):
            p = batch.problem(i)
            Ls.append(p.L_dense().reshape(-1))
            errs.append(p.info()["rel_err"])
        return {"L": torch.cat(Ls), "rel_err": torch.tensor(errs)}
    if kind == "gradient":
        return G.backward(state["X"], state["A1"], case["T"], state["supports"], gL=state["gL"])
    ctx = state["ctx"]
    ctx.reset()
    rel = ctx.iterate(case["iters"])
    return {"W": ctx.W(), **_results(ctx, rel)}


# ---- work -----------------------------------------------------------------------------------
def _solve_work(m, n, r, q, k, iters):
    """Iterations of Algorithm 1: each of the 6q+3 products and the S-step needs the matrix
    once (it is larger than any on-chip memory, and every product needs the whole of the one
    before it), and each product its skinny operands; L and S are written once at the end."""
    p = 6 * q + 3
    return {"bytes": iters * ((p + 1) * 4.0 * m * n + p * 4.0 * (m + n) * r + 12.0 * k) + 4.0 * m * n + 12.0 * k,
            "flops": iters * (p + 1) * 2.0 * m * n * r + 2.0 * m * n * r}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        tot = {"bytes": 0.0, "flops": 0.0}
        for m, n, r, density in _batch_shapes(case):
            w = _solve_work(m, n, r, 1, density * m * n, case["iters"])
            tot = {key: tot[key] + w[key] for key in tot}
        return tot
    m, n = case["m"], case["n"]
    mn = float(m) * n
    if kind == "product":
        return {"bytes": 4.0 * mn + 4.0 * (m + n) * case["r"], "flops": 2.0 * mn * case["r"]}
    if kind == "threshold":
        return {"bytes": 4.0 * mn + 12.0 * case["density"] * mn, "flops": 0.0}
    if kind in ("solve", "once"):
        return _solve_work(m, n, case["r"], case["q"], case["density"] * mn, case["iters"])
    if kind == "gradient":
        T, r, k = case["T"], case["r"], case["density"] * mn
        # X and the dense gradient read once, dX written once, and per unrolled iteration five
        # products with the iterate and one rank-3r accumulation
        return {"bytes": 12.0 * mn + 8.0 * (T - 1) * k + T * 5 * 4.0 * mn, "flops": T * (5 * 2.0 + 6.0) * mn * r}
    d, r, it = case["d"], case["r"], case["iters"]
    return {"bytes": it * (2 * 4.0 * mn + 12.0 * case["density"] * mn) + 4.0 * mn,
            "flops": it * (2.0 * mn * d + 2.0 * mn * r) + 2.0 * mn * r}


# ---- the same in 64 bits ----------------------------------------------------------------------
def _qr(A):
    Q, R = torch.linalg.qr(A)
    return Q, R


def _topk_support(R, k):
    """Ascending positions of the k largest |R| (ties by position)."""
    return torch.topk(R.abs().reshape(-1), k, sorted=False).indices.sort().values


def _lstep64(Z, A1, q):
    B = A1
    for i in range(4 * q + 2):
        B, _ = _qr(Z @ B if i % 2 == 0 else Z.T @ B)
    Q2 = B
    Q, M = _qr(Z @ Q2)
    for i in range(1, 2 * q + 1):
        Q, Rf = _qr(Z.T @ Q if i % 2 == 1 else Z @ Q)
        M = Rf @ M
    Um, s, Vh = torch.linalg.svd(M)
    return Q @ Um, s ** (1.0 / (2 * q + 1)), Q2 @ Vh.T


def _refine64(Z, U, V):
    """The precision form's correction: the tangent-space projection of Z at (U, V),
    P_U Z + Z P_V - P_U Z P_V, truncated to the rank of U."""
    r = U.shape[1]
    A, B = Z @ V, Z.T @ U
    Qa, Ra = _qr(torch.cat([U, A], 1))
    Qb, Rb = _qr(torch.cat([V, B], 1))
    C = U.T @ A
    K = torch.zeros(2 * r, 2 * r, dtype=Z.dtype, device=Z.device)
    K[:r, :r] = -C
    K[:r, r:] = torch.eye(r, dtype=Z.dtype, device=Z.device)
    K[r:, :r] = torch.eye(r, dtype=Z.dtype, device=Z.device)
    Uc, s, Vch = torch.linalg.svd(Ra @ K @ Rb.T)
    return Qa @ Uc[:, :r], s[:r], Qb @ Vch[:r].T


def _solve64(X, A1, k, q, iters, half=False):
    X, A1 = X.double(), A1.double()
    Z = X.clone()
    for _ in range(iters):
        U, s, V = _lstep64(Z, A1, q)
        if half:
            U, s, V = _refine64(Z, U, V)
        L = (U * s) @ V.T
        R = X - L
        idx = _topk_support(R, k)
        val = R.view(-1)[idx]
        Z.copy_(X)
        Z.view(-1)[idx] = L.view(-1)[idx]
    R.view(-1)[idx] = 0.0
    return L, idx, val, float((R.square().sum() / X.square().sum()).item())


def _gradient64(X, A1, supports, gL):
    X = X.double().requires_grad_(True)
    A1 = A1.double()
    Z = X
    for t in range(len(supports) + 1):
        Q, _ = _qr(Z.T @ (Z @ A1))
        L = (Z @ Q) @ Q.T
        if t < len(supports):
            M = torch.zeros(X.numel(), dtype=torch.bool, device="cuda")
            M[supports[t]] = True
            Z = torch.where(M.view_as(X), L, X)
    (L * gL.double()).sum().backward()
    return X.grad


def _lingodec64(X, F, r, lam, iters):
    X, F = X.double(), F.double()
    Qf, Rf = _qr(F)
    S = torch.zeros_like(X)
    for _ in range(iters):
        Uy, s, Vh = torch.linalg.svd((X - S) @ Qf, full_matrices=False)
        M = (Uy[:, :r] * s[:r]) @ Vh[:r]
        W = torch.linalg.solve_triangular(Rf, M.T, upper=True).T
        L = W @ F.T
        R = X - L
        S = R.sign() * (R.abs() - lam).clamp_min(0.0)
    idx = S.reshape(-1).nonzero().reshape(-1)
    rel = ((R - S).square().sum() / X.square().sum()).item()
    return W, L, idx, S.reshape(-1)[idx], float(rel)


def exact(case, seed):
    kind, s = case["kind"], _inputs(case, seed)
    if kind == "product":
        Z, B = s["Z"].double(), s["B"].double()
        return Z.T @ B if case["trans"] else Z @ B
    if kind == "threshold":
        R = s["R"].double()
        idx = _topk_support(R, s["k"])
        return idx, R.view(-1)[idx]
    if kind in ("solve", "once"):
        L, idx, val, rel = _solve64(s["X"], s["A1"], s["k"], case["q"], case["iters"], case["half"])
        return {"L": L, "S_idx": idx, "S_val": val, "rel_err": rel}
    if kind == "batch":
        got = [_solve64(X, A1, k, 1, case["iters"]) for X, A1, k in zip(s["Xs"], s["A1s"], s["ks"])]
        return {"L": torch.cat([L.reshape(-1) for L, _, _, _ in got]),
                "rel_err": torch.tensor([e for _, _, _, e in got])}
    if kind == "gradient":
        return _gradient64(s["X"], s["A1"], s["supports"], s["gL"])
    W, L, idx, val, rel = _lingodec64(s["X"], s["F"], case["r"], s["lam"], case["iters"])
    return {"W": W, "L": L, "S_idx": idx, "S_val": val, "rel_err": rel}
