"""Workloads of the HPR-QP library, each one pass through its public entry points.

A case stands for one thing that a program has the library do: a solve of one problem (from the
origin, from a neighbouring solution, or together with the creation of its handle from host
arrays), a batch of independent problems, the learned start's inference and training, and the
tensor-core product below them.  Solves run a fixed budget of inner steps, as a program with a
deadline would ask for; a problem that meets its tolerance earlier stops earlier.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2507_02470_gb300 as hp
from paper_2507_02470_gb300 import learned

TOL = 1e-8
L2_BYTES = 100e6          # a working set below this stays in the GPU's cache between inner steps
INF = float("inf")


def listed():
    return [
        # the small plain problem (A 1 % dense, Q = M^T M): latency and launches are everything
        {"name": "solve_small", "kind": "cqp", "n": 1000, "m": 500, "a_row": 10, "q": "factor", "iters": 1000},
        # a member of a parametric family, started from its neighbour's solution
        {"name": "resolve_family", "kind": "family", "n": 100_000, "m": 50_000, "a_row": 6, "q": "sum", "iters": 300},
        # one large sparse problem from the origin, power method included
        {"name": "solve_large", "kind": "cqp", "n": 1_000_000, "m": 500_000, "a_row": 6, "q": "sum", "iters": 500},
        # explicit Q (so preconditioned), odd sizes: handle made from host arrays, solve, results read back
        {"name": "once_csr", "kind": "once", "n": 20_011, "m": 7_003, "a_row": 5, "q": "csr", "iters": 1250},
        # Lasso: no rows, l1 term, one large matrix-free factor
        {"name": "solve_lasso", "kind": "lasso", "p": 50_000, "q": 500_000, "row": 250, "iters": 300},
        # QAP relaxation, Q applied as dense d x d products
        {"name": "solve_qap", "kind": "qap", "d": 256, "iters": 200},
        # one portfolio problem with a dense factor
        {"name": "solve_portfolio", "kind": "portfolio", "n": 4001, "iters": 500},
        # many portfolio problems of mixed sizes
        {"name": "batch_mixed", "kind": "batch", "count": 400, "lo": 50, "hi": 5000, "iters": 300},
        # many small portfolio problems
        {"name": "batch_small", "kind": "batch", "count": 700, "lo": 30, "hi": 600, "iters": 500},
        # learned start: inference for a batch of members
        {"name": "predict", "kind": "predict", "n": 100_000, "m": 50_000, "B": 256},
        # learned start: a few optimiser steps of its network, then the weights read back
        {"name": "train", "kind": "train", "d0": 512, "hidden": 1024, "out": 257, "B": 256, "steps": 24},
        # learned start: the feature projection of a block of members
        {"name": "project", "kind": "project", "M": 512, "N": 1500, "K": 150_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cqp", "cqp", "family", "once", "lasso", "qap", "portfolio", "batch", "predict", "train",
                       "project"])
    if kind in ("cqp", "family", "once"):
        n = _log(rng, 150, 400_000 if kind != "once" else 60_000)
        return {"kind": kind, "n": n, "m": max(1, int(n * rng.uniform(0.1, 0.8))), "a_row": rng.randint(2, 12),
                "q": rng.choice(["factor", "sum", "csr"] if n <= 20_000 else ["sum", "csr"]),
                "iters": rng.choice([100, 200, 300, 330, 450])}
    if kind == "lasso":
        q = _log(rng, 3000, 300_000)
        return {"kind": kind, "p": max(50, int(q * rng.uniform(0.05, 0.3))), "q": q, "row": rng.randint(20, 200),
                "iters": rng.choice([100, 150, 200])}
    if kind == "qap":
        return {"kind": kind, "d": rng.randint(12, 256), "iters": rng.choice([100, 120, 200])}
    if kind == "portfolio":
        return {"kind": kind, "n": _log(rng, 60, 5000), "iters": rng.choice([100, 300, 420])}
    if kind == "batch":
        lo = _log(rng, 30, 1000)
        return {"kind": kind, "count": _log(rng, 20, 400), "lo": lo, "hi": min(4000, lo * rng.randint(2, 8)),
                "iters": rng.choice([100, 200, 300])}
    if kind == "predict":
        n = _log(rng, 2000, 100_000)
        return {"kind": kind, "n": n, "m": int(n * rng.uniform(0.2, 0.6)) + 1, "B": _log(rng, 1, 256)}
    if kind == "train":
        return {"kind": kind, "d0": 8 * rng.randint(8, 64), "hidden": 8 * rng.randint(16, 128),
                "out": 1 + _log(rng, 16, 256), "B": _log(rng, 16, 256), "steps": rng.randint(8, 24)}
    return {"kind": kind, "M": rng.randint(64, 512), "N": _log(rng, 1, 1500), "K": _log(rng, 2000, 150_000)}


# ---------------------------------------------------------------------------------- problems
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _uniform(g, n, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _normal(g, n):
    return torch.randn(n, generator=g, device="cuda", dtype=torch.float64)


def _sparse(g, rows, cols, per_row, scale=1.0):
    """Uniform random pattern with about `per_row` entries a row, N(0, scale) values: CSR tensors."""
    keys = torch.randint(0, rows * cols, (rows * per_row,), generator=g, device="cuda", dtype=torch.int64)
    keys = torch.unique(keys)
    return _csr(keys // cols, keys % cols, _normal(g, keys.numel()) * scale, rows)


def _csr(r, c, v, rows):
    """CSR arrays of entries that are sorted by row."""
    rp = torch.zeros(rows + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(r, minlength=rows), 0)
    return rp.to(torch.int32), c.to(torch.int32), v


def _coo(M):
    rp, c, v = M
    cnt = (rp[1:] - rp[:-1]).to(torch.int64)
    return torch.repeat_interleave(torch.arange(cnt.numel(), device=v.device), cnt), c.to(torch.int64), v


def _mul(M, x):
    """M x for CSR arrays."""
    r, c, v = _coo(M)
    return torch.zeros(M[0].numel() - 1, dtype=torch.float64, device=v.device).index_add_(0, r, v * x[c])


def _term(kind, p=0, csr=(None, None, None), offsets=None, diags=None, dense=None):
    return SimpleNamespace(kind=kind, p=p, rowptr=csr[0], colidx=csr[1], vals=csr[2], offsets=offsets, diags=diags,
                           dense=dense)


def _problem(n, m, A, c, l, u, L, U, phi, lam, terms):
    return SimpleNamespace(n=n, m=m, A_rowptr=A[0], A_colidx=A[1], A_vals=A[2], c=c, l=l, u=u, L=L, U=U, phi=phi,
                           lam=lam, qterms=terms)


def _cqp(case, seed):
    """Sparse problem with box [-5, 5] (factor Q: [0, 10]): 30 % equality rows, the rest one-sided,
    feasible by construction; Q a factor, a band plus a thin factor, or that sum as one matrix."""
    g = _gen(seed)
    n, m = case["n"], case["m"]
    A = _sparse(g, m, n, case["a_row"])
    c = _normal(g, n)
    x0 = _uniform(g, n)
    Ax = _mul(A, x0)
    u = Ax + _uniform(g, m)
    l = torch.full_like(u, -INF)
    eq = max(1, int(0.3 * m))
    l[:eq] = Ax[:eq]
    u[:eq] = Ax[:eq]
    if case["q"] == "factor":
        p = max(2, n // 10)
        terms = [_term("factor", p, _sparse(g, p, n, max(3, n // 50)))]
        lo, hi = 0.0, 10.0
    else:
        d = torch.zeros(3, n, dtype=torch.float64, device="cuda")
        d[0] = _uniform(g, n, 1.0, 2.0)
        d[1, :n - 1] = _uniform(g, n - 1, -0.2, 0.2)
        d[2, :n - 2] = _uniform(g, n - 2, -0.2, 0.2)
        s = max(1, n // 100)
        S = _sparse(g, s, n, 3)
        lo, hi = -5.0, 5.0
        if case["q"] == "sum":
            off = torch.tensor([0, 1, 2], dtype=torch.int32)
            terms = [_term("dia", offsets=off, diags=d), _term("factor", s, S)]
        else:
            terms = [_term("csr", csr=_assemble(n, d, S))]
    L, U = (torch.full((n,), v, dtype=torch.float64, device="cuda") for v in (lo, hi))
    return _problem(n, m, A, c, l, u, L, U, 0, 0.0, terms)


def _assemble(n, d, S):
    """Band d (offsets 0, 1, 2, mirrored) + S^T S as CSR arrays."""
    i = torch.arange(n, device="cuda")
    r, c, v = [i], [i], [d[0]]
    for o in (1, 2):
        r += [i[:n - o], i[o:]]
        c += [i[o:], i[:n - o]]
        v += [d[o, :n - o], d[o, :n - o]]
    rp, sc, sv = S[0].to(torch.int64), S[1].to(torch.int64), S[2]
    cnt = rp[1:] - rp[:-1]
    for a in range(int(cnt.max())):
        for b in range(int(cnt.max())):
            has = (cnt > a) & (cnt > b)
            ka, kb = rp[:-1][has] + a, rp[:-1][has] + b
            r.append(sc[ka])
            c.append(sc[kb])
            v.append(sv[ka] * sv[kb])
    key, inv = torch.unique(torch.cat(r) * n + torch.cat(c), return_inverse=True)
    val = torch.zeros(key.numel(), dtype=torch.float64, device="cuda").index_add_(0, inv, torch.cat(v))
    return _csr(key // n, key % n, val, n)


def _lasso(case, seed):
    g = _gen(seed)
    p, q = case["p"], case["q"]
    B = _sparse(g, p, q, case["row"], 1.0 / math.sqrt(p))
    xs = torch.zeros(q, dtype=torch.float64, device="cuda")
    k = max(1, q // 100)
    xs[torch.randperm(q, generator=g, device="cuda")[:k]] = _normal(g, k)
    b = _mul(B, xs) + 0.01 * _normal(g, p)
    r, cidx, v = _coo(B)
    c = -torch.zeros(q, dtype=torch.float64, device="cuda").index_add_(0, cidx, v * b[r])
    e = torch.zeros(0, dtype=torch.float64, device="cuda")
    A = (torch.zeros(1, dtype=torch.int32, device="cuda"), e.to(torch.int32), e)
    inf = torch.full((q,), INF, dtype=torch.float64, device="cuda")
    return _problem(q, 0, A, c, e, e, -inf, inf, 1, 0.1 * float(c.abs().max()), [_term("factor", p, B)])


def _qap(case, seed):
    """The relaxation of a quadratic assignment: flows, Manhattan distances of random points, and a
    feasible pair (s, t) of the eigenvalue bound, which keeps Q positive semidefinite."""
    g = _gen(seed)
    d = case["d"]
    F = torch.randint(0, 10, (d, d), generator=g, device="cuda").double()
    F = torch.triu(F * (torch.rand(d, d, generator=g, device="cuda") < 0.6), 1)
    F = F + F.T
    side = max(2, math.isqrt(d) + 2)
    pt = torch.randint(0, side, (d, 2), generator=g, device="cuda")
    D = (pt[:, None, :] - pt[None, :, :]).abs().sum(2).double()
    al, VA = torch.linalg.eigh(F)
    be, VB = torch.linalg.eigh(D)
    ab = al[:, None] * be[None, :]
    s = ab.amin(1)
    t = (ab - s[:, None]).amin(0)
    S = VA @ torch.diag(s) @ VA.T
    T = VB @ torch.diag(t) @ VB.T
    dense = torch.cat([2.0 * F, D, S + S.T, T + T.T]).reshape(-1).contiguous()
    n = d * d
    i = torch.arange(n, device="cuda")
    rows = torch.cat([i // d, d + i // d])
    cols = torch.cat([(i % d) * d + i // d, i])
    cols[:n] = cols[:n].reshape(d, d).sort(1).values.reshape(-1)
    one = lambda k, v=1.0: torch.full((k,), v, dtype=torch.float64, device="cuda")  # noqa: E731
    return _problem(n, 2 * d, _csr(rows, cols, one(2 * n), 2 * d), one(n, 0.0), one(2 * d), one(2 * d), one(n, 0.0),
                    one(n, INF), 0, 0.0, [_term("qap", d, dense=dense)])


def _portfolio(n, g):
    """Factor model with a budget row and ten sector rows, weights in [0, 0.1]."""
    k, sectors = max(5, n // 20), 10
    F = torch.randn(k, n, generator=g, device="cuda", dtype=torch.float64) / math.sqrt(n)
    d = _uniform(g, n, 0.01, 0.1)
    sector = torch.randperm(n, generator=g, device="cuda") % sectors
    at = torch.sort(sector, stable=True).indices
    rows = torch.cat([torch.zeros(n, dtype=torch.int64, device="cuda"), 1 + sector[at]])
    cols = torch.cat([torch.arange(n, device="cuda"), at])
    l = torch.full((11,), -INF, dtype=torch.float64, device="cuda")
    u = torch.full((11,), 0.3, dtype=torch.float64, device="cuda")
    l[0] = u[0] = 1.0
    c = 0.1 * _normal(g, n)
    A = _csr(rows, cols, torch.ones(2 * n, dtype=torch.float64, device="cuda"), 11)
    return _problem(n, 11, A, c, l, u, torch.zeros_like(c), torch.full_like(c, 0.1), 0, 0.0,
                    [_term("dense_factor", k, dense=F), _term("diag", dense=d)])


def _batch_sizes(case):
    """The sizes of a batch: spread evenly over its range, so that every seed asks for the same work."""
    k = case["count"]
    return [int(round(case["lo"] + (case["hi"] - case["lo"]) * ((i * 0.6180339887498949) % 1.0))) for i in range(k)]


def _to_host(p):
    """The same problem in host memory."""
    def h(v):
        return v.cpu().numpy() if isinstance(v, torch.Tensor) else v

    q = SimpleNamespace(**{k: h(v) for k, v in vars(p).items() if k != "qterms"})
    q.qterms = [SimpleNamespace(**{k: h(v) for k, v in vars(t).items()}) for t in p.qterms]
    return q


def _make(case, seed):
    kind = case["kind"]
    if kind == "lasso":
        return _lasso(case, seed)
    if kind == "qap":
        return _qap(case, seed)
    if kind == "portfolio":
        return _portfolio(case["n"], _gen(seed))
    return _cqp(case, seed)


def _member(p, g):
    """The next member of a family: other costs and looser inequality rows."""
    c = p.c + 0.1 * _normal(g, p.n)
    u = torch.where(torch.isinf(p.l), p.u + 0.1 * _uniform(g, p.m), p.u)
    return c, u


# ---------------------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        g = _gen(seed)
        probs = [_to_host(_portfolio(n, g)) for n in _batch_sizes(case)]
        return {"case": case, "batch": hp.BatchSolver(probs)}
    if kind == "predict":
        n, m, B = case["n"], case["m"], case["B"]
        rng = np.random.default_rng(seed)
        ws = learned.LearnedWarmStart(n, m, np.full(n, -5.0), np.full(n, 5.0), np.full(m, -np.inf), np.zeros(m),
                                      max_batch=256, seed=seed % 1000)
        g = _gen(seed)
        N = 64
        C0, U0 = _normal(g, n), _normal(g, m)

        def members(k):
            return (C0 + 0.1 * _normal(g, k * n).reshape(k, n), U0 + 0.1 * _uniform(g, k * m).reshape(k, m))

        data = members(N)
        Z = 0.5 * _normal(g, n + m) + 0.1 * _normal(g, N * (n + m)).reshape(N, n + m)
        ws.fit(data, Z, np.exp(rng.normal(0.0, 0.3, N)), epochs=1, batch=32)
        Cs, Us = members(B)
        return {"case": case, "ws": ws, "C": Cs, "U": Us}
    if kind == "train":
        rng = np.random.default_rng(seed)
        dims = [case["d0"], case["hidden"], case["hidden"], case["out"]]
        net = learned.MLP(dims, case["B"], stream=torch.cuda.current_stream())
        for i in range(3):
            net.set_layer(i, rng.standard_normal((dims[i + 1], dims[i])) * math.sqrt(2.0 / dims[i]),
                          0.1 * rng.standard_normal(dims[i + 1]))
        g = _gen(seed)
        X = torch.randn(case["B"], dims[0], generator=g, device="cuda").bfloat16()
        dY = [torch.randn(case["B"], dims[3], generator=g, device="cuda") / case["B"] for _ in range(2)]
        return {"case": case, "net": net, "X": X, "dY": dY}
    if kind == "project":
        g = _gen(seed)
        M, N, K = case["M"], case["N"], case["K"]
        P = torch.randn(M, K, generator=g, device="cuda") / math.sqrt(K)
        return {"case": case, "P": learned.cast_bf16(P), "V": _normal(g, N * K).reshape(N, K)}
    p = _make(case, seed)
    if kind == "once":
        return {"case": case, "host": _to_host(p)}
    st = {"case": case, "solver": hp.Solver(p)}
    st["out"] = [torch.empty(k, dtype=torch.float64, device="cuda") for k in (p.n, p.m, p.n, p.n)]
    if kind == "family":
        s = st["solver"]
        s.solve(tol=TOL, max_iter=300)
        x, y, _, _, k = s.get()
        s.set_lambda(k["lambda_A"], k["lambda_Q"])
        st["start"] = [torch.from_numpy(v).cuda() for v in (x, y)]
        st["member"] = _member(p, _gen(seed + 1_000_003))
    return st


# ---------------------------------------------------------------------------------- run
def _solution(x, y, z, w, k):
    return {"x": x, "y": y, "z": z, "w": w, "pobj": k["pobj"], "iters": k["iters"]}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        b = state["batch"]
        b.solve(tol=TOL, max_iter=case["iters"])
        got = [b.get(i) for i in range(b.count)]
        return {"x": np.concatenate([r[0] for r in got]), "y": np.concatenate([r[1] for r in got]),
                "z": np.concatenate([r[2] for r in got]), "pobj": np.array([r[3]["pobj"] for r in got]),
                "iters": np.array([r[3]["iters"] for r in got])}
    if kind == "predict":
        Z0, sigma0 = state["ws"].predict(state["C"], state["U"])
        return {"Z0": Z0, "sigma0": sigma0}
    if kind == "train":
        net = state["net"]
        for i in range(case["steps"]):
            Y = net.forward(state["X"])
            net.backward(state["dY"][i % 2])
            net.adam(lr=1e-4)
        return {"Y": Y, "layers": [net.get_layer(i) for i in range(3)]}
    if kind == "project":
        return {"F": learned.gemm_bf16(state["P"], learned.cast_bf16(state["V"]))}
    if kind == "once":
        with hp.Solver(state["host"]) as s:
            s.solve(tol=TOL, max_iter=case["iters"])
            return _solution(*s.get())
    s = state["solver"]
    if kind == "family":
        s.set_data(c=state["member"][0], u=state["member"][1])
        s.set_warm_start(*state["start"])
    s.solve(tol=TOL, max_iter=case["iters"])
    return _solution(*s.get(*state["out"]))


# ---------------------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind == "project":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2.0 * M * K + 8.0 * N * K + 4.0 * M * N, "flops": 2.0 * M * N * K}
    if kind == "predict":
        D, B = case["n"] + case["m"], case["B"]
        net = 512 * 1024 + 1024 * 1024 + 1024 * 257
        return {"bytes": 2.0 * D * (512 + 256) + 2.0 * net + 16.0 * D * B, "flops": 2.0 * B * (D * (512 + 256) + net)}
    if kind == "train":
        net = case["d0"] * case["hidden"] + case["hidden"] ** 2 + case["hidden"] * case["out"]
        # forward, two backward products, and the optimiser's weights and two moments each way
        return {"bytes": case["steps"] * 24.0 * net, "flops": case["steps"] * 6.0 * case["B"] * net}
    it = case["iters"]
    if kind == "batch":
        data = flops = 0.0
        for n in _batch_sizes(case):
            k = max(5, n // 20)
            data += 8.0 * n * (k + 40)
            flops += it * n * (4.0 * k + 90.0)
        return {"bytes": data * it if data > L2_BYTES else data, "flops": flops}
    if kind == "lasso":
        n, m, nnz = case["q"], 0, 0
        qb, qf = 12.0 * case["p"] * case["row"], 4.0 * case["p"] * case["row"]
    elif kind == "qap":
        n, m, nnz = case["d"] ** 2, 2 * case["d"], 2 * case["d"] ** 2
        qb, qf = 32.0 * n, 8.0 * case["d"] ** 3
    elif kind == "portfolio":
        n, m, nnz = case["n"], 11, 2 * case["n"]
        qb, qf = 8.0 * n * (max(5, n // 20) + 1), 4.0 * n * max(5, n // 20)
    else:
        n, m = case["n"], case["m"]
        nnz = m * case["a_row"]
        f = max(2, n // 10) * max(3, n // 50) if case["q"] == "factor" else 3 * max(1, n // 100)
        qb, qf = (12.0 * f, 4.0 * f) if case["q"] == "factor" else (24.0 * n + 12.0 * f, 10.0 * n + 4.0 * f)
    # each stored matrix once, and the vectors that the step carries on from one to the next
    step = 12.0 * nnz + qb + 8.0 * (14 * n + 5 * m)
    return {"bytes": step * it if step > L2_BYTES else step,
            "flops": it * (4.0 * nnz + (1 if m == 0 else 2) * qf + 40.0 * n + 12.0 * m)}


# ---------------------------------------------------------------------------------- exact
def exact(case, seed):
    kind = case["kind"]
    if kind == "project":
        g = _gen(seed)
        M, N, K = case["M"], case["N"], case["K"]
        P = (torch.randn(M, K, generator=g, device="cuda") / math.sqrt(K)).bfloat16().double()
        V = _normal(g, N * K).reshape(N, K).float().bfloat16().double()
        return {"F": P @ V.T}
    if kind in ("batch", "predict", "train"):
        return None          # long runs of their own, or whose 16-bit roundings have no 64-bit value
    p = _make(case, seed)
    if kind == "family":
        x, y, _, _, _, _, lam = _hpr(p, 300)
        p.c, p.u = _member(p, _gen(seed + 1_000_003))
        got = _hpr(p, case["iters"], x, y, lam)
    else:
        got = _hpr(p, case["iters"])
    return dict(zip(("x", "y", "z", "w", "pobj", "iters"), (*got[:5], None)))


def _scaling(p):
    """Ten Ruiz passes and a Pock-Chambolle pass on [Q A^T; A 0], for one explicit Q in a box."""
    n = p.n
    ar, ac, av = _coo((p.A_rowptr, p.A_colidx, p.A_vals))
    qr, qc, qv = _coo((p.qterms[0].rowptr, p.qterms[0].colidx, p.qterms[0].vals))
    r, c, v = torch.cat([qr, n + ar, ac]), torch.cat([qc, ac, n + ar]), torch.cat([qv, av, av]).abs()
    s = torch.ones(n + p.m, dtype=torch.float64, device="cuda")
    for i in range(11):
        norm = torch.zeros_like(s)
        norm.scatter_reduce_(0, c, v * s[r] * s[c], "amax" if i < 10 else "sum")
        s = torch.where(norm > 0, s / norm.sqrt(), s)
    return s[:n], s[n:]


def _hpr(p, iters, x0=None, y0=None, lam=None):
    """Algorithm 4 of the paper in plain 64-bit torch: (x, y, z, w, objective, steps, (lambda_A, lambda_Q))."""
    n, m = p.n, p.m
    ar, ac, av = _coo((p.A_rowptr, p.A_colidx, p.A_vals))
    c, l, u, L, U = p.c, p.l, p.u, p.L, p.U
    d, e = torch.ones_like(c), torch.ones(m, dtype=torch.float64, device="cuda")
    if p.phi == 0 and p.qterms[0].kind == "csr":
        d, e = _scaling(p)
        av = av * e[ar] * d[ac]
        c, l, u, L, U = c * d, l * e, u * e, L / d, U / d

    def mat(r, cidx, v, rows, x):
        return torch.zeros(rows, dtype=torch.float64, device="cuda").index_add_(0, r, v * x[cidx])

    A = lambda x: mat(ar, ac, av, m, x)      # noqa: E731
    AT = lambda y: mat(ac, ar, av, n, y)     # noqa: E731
    ops = []
    for t in p.qterms:
        if t.kind == "csr":
            r, k, v = _coo((t.rowptr, t.colidx, t.vals))
            ops.append(lambda x, r=r, k=k, v=v * d[r] * d[k]: mat(r, k, v, n, x))
        elif t.kind == "factor":
            r, k, v = _coo((t.rowptr, t.colidx, t.vals))
            ops.append(lambda x, r=r, k=k, v=v, q=t.p: mat(k, r, v, n, mat(r, k, v, q, x)))
        elif t.kind == "dense_factor":
            ops.append(lambda x, F=t.dense.reshape(t.p, n): F.T @ (F @ x))
        elif t.kind == "diag":
            ops.append(lambda x, g=t.dense: g * x)
        elif t.kind == "dia":
            def band(x, b=t.diags):
                y = b[0] * x
                for o in (1, 2):
                    y[:n - o] += b[o, :n - o] * x[o:]
                    y[o:] += b[o, :n - o] * x[:n - o]
                return y
            ops.append(band)
        else:
            def qap(x, M=t.dense.reshape(4, t.p, t.p)):
                X = x.reshape(M.shape[1], M.shape[1]).T
                return (M[0] @ X @ M[1] - M[2] @ X - X @ M[3]).T.reshape(-1)
            ops.append(qap)
    Q = lambda x: sum(f(x) for f in ops)     # noqa: E731

    def power(f, dim):
        v = 0.5 + ((torch.arange(1, dim + 1, device="cuda") * 2654435761) % (1 << 32)).double() / 4294967296.0
        v, last = v / v.norm(), 0.0
        for k in range(5000):
            w = f(v)
            got = float(v @ w)
            v = w / w.norm()
            if k and abs(got - last) <= 1e-6 * abs(got):
                return 1.01 * got
            last = got
        return 1.01 * got

    lA, lQ = lam or (power(lambda y: A(AT(y)), m) if m else 0.0, power(Q, n))
    fin = lambda v: torch.where(torch.isfinite(v), v.abs(), torch.zeros_like(v))   # noqa: E731
    b, b0 = torch.maximum(fin(l), fin(u)), torch.maximum(fin(p.l), fin(p.u))
    nb, nc = float(b.norm()), float(c.norm())
    sg = nb / nc if 1e-16 <= nb <= 1e16 and 1e-16 <= nc <= 1e16 else 1.0
    top = lambda v: float(v.max()) if v.numel() else 0.0   # noqa: E731
    bmax, cmax = top(b0), float(p.c.abs().max())
    x = torch.zeros_like(c) if x0 is None else x0 / d
    y = torch.zeros_like(l) if y0 is None else y0 / e
    w = x.clone()
    ax, ay, aw = x, y, w
    k = t = r = 0
    a3, first, before, start = 0.5, 0.0, 0.0, 0.0
    while True:
        Qw, ATy = Q(w), AT(y)
        rz = x + sg * (ATy - c - Qw)
        xb = rz if p.phi == 0 else torch.sign(rz) * torch.clamp(rz.abs() - sg * p.lam, min=0.0)
        xb = torch.minimum(torch.maximum(xb, L), U)
        z = (xb - rz) / sg
        xh = 2 * xb - x
        wb = (xh + sg * lQ * w) / (1 + sg * lQ)
        s = sg / (1 + sg * lQ)
        yb, ATyb = y, ATy
        if m:
            ry = A(xh + sg * (Qw - Q(wb))) - sg * lA * y
            yb = (torch.minimum(torch.maximum(ry, l), u) - ry) / (sg * lA)
            ATyb = AT(yb)
            wb = wb + s * (ATyb - ATy)
        k += 1
        if k % 100 == 0 or k >= iters:
            Qx, Ax = Q(xb), A(xb)
            dual = lambda v, lo, hi: torch.where(v > 0, lo * v, torch.where(v < 0, hi * v, torch.zeros_like(v))).sum()  # noqa: E731
            obj = float(0.5 * (xb @ Qx) + c @ xb + p.lam * xb.abs().sum())
            dobj = float(-0.5 * (xb @ Qx) + dual(yb, l, u) - (dual(-z, U, L) if p.phi == 0 else 0.0))
            ep = top(((Ax - torch.minimum(torch.maximum(Ax, l), u)) / e).abs()) / (1 + max(bmax, top((Ax / e).abs())))
            ed = top(((ATyb - Qx + z - c) / d).abs()) / (1 + max(cmax, top((ATyb / d).abs()), top((Qx / d).abs())))
            if max(ep, ed, abs(obj - dobj) / (1 + max(abs(obj), abs(dobj)))) <= TOL or k >= iters:
                return xb * d, yb * e, z / d, wb * d, obj, k, (lA, lQ)
        restart = False
        if t == 0 or k % 10 == 0:
            dx, dy, dw = x - xb, y - yb, w - wb
            Qdw, Ady = Q(dw), ATy - ATyb
            th1 = lA * float(dy @ dy) + lQ * float(dw @ Qdw) - 2 * float(Qdw @ Ady)
            R2 = sg * th1 + float(dx @ dx) / sg + sg * s * float(Ady @ Q(Ady)) + 2 * float(dx @ (Ady - Qdw))
            R = math.sqrt(max(R2, 0.0))
            if t == 0:
                start = R
            else:
                restart = R <= 0.2 * start or (R <= 0.8 * start and R > before) or t + 1 >= a3 * k
            before = R
        if not restart:
            t += 1
            f = 1.0 / (t + 1)
            x, y, w = (f * o + (1 - f) * (2 * bar - v) for o, bar, v in ((ax, xb, x), (ay, yb, y), (aw, wb, w)))
            continue
        first = R if r == 0 else first
        ratio = R / first if first > 0 else 0.0
        a3 = 0.2 if ratio <= 0.1 else a3
        dx, dy, dw = xb - ax, yb - ay, wb - aw
        Qdw, Ady = Q(dw), AT(dy)
        th1 = max(lA * float(dy @ dy) + lQ * float(dw @ Qdw) - 2 * float(Qdw @ Ady), 1e-12)
        th2, th3 = max(float(dx @ dx), 1e-12), float(Ady @ Q(Ady))
        lo = hi = math.sqrt(th2 / th1)
        if th3 > 0 and lQ > 0:
            lo = math.sqrt(th2 / (th1 + th3 / lQ))
            for _ in range(200):
                mid = 0.5 * (lo + hi)
                up = th1 - th2 / mid ** 2 + th3 * mid * (2 + lQ * mid) / (1 + lQ * mid) ** 2 > 0
                lo, hi = (lo, mid) if up else (mid, hi)
                if hi - lo <= 4e-16 * hi:
                    break
        beta = math.exp(-ratio)
        sg = math.exp(beta * math.log(0.5 * (lo + hi)) + (1 - beta) * math.log(sg))
        x, y, w = xb, yb, wb
        ax, ay, aw = x, y, w
        t, r = 0, r + 1
