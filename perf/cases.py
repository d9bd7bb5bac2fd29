"""Measured cases: what a user of this package has it do, through gsi.Solver,
gsi.Batch and gsi.MLP, from the smallest grid to the 128^3 one.

A solver pass starts from a new block (`reset`), runs a fixed number of
iterations and fetches the basis, so that it does the same work on every call
and its outputs can be compared (a whole solve repeats the same iterations
hundreds of times). Start blocks, graphs and dense operators come from the
seed."""
import math

import numpy as np
import torch

from paper_2306_10379_gb300 import gsi

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # The plain float64 gradient method on a 32 x 32 Dirichlet grid: the
        # first thing anyone runs, and the smallest call (launches and host
        # round trips).
        _fd("fd2d_32_p8_f64_sd", (32, 32), 8, 10, method="sd", precision="f64"),
        # The same grid with the default arithmetic and conjugate gradients,
        # and its Ritz values at the end, as a finished solve fetches them.
        _fd("fd2d_32_p8_cg", (32, 32), 8, 10, evals=True),
        # The FD3D matrix of the paper's method comparison (n = 35,000), its
        # narrow and its wide block; largest and smallest eigenvalues.
        _fd("fd3d_35k_p16_cg", (35, 40, 25), 16, 10),
        _fd("fd3d_35k_p64_min_cg", (35, 40, 25), 64, 10, which=-1),
        # A ragged graph operator in SELL-32 with an odd block width: rows of
        # uneven length, n no multiple of anything, blocks off 16 bytes.
        {"name": "graph_sell_p33_cg", "kind": "solve", "op": "er", "n": 50021, "p": 33, "steps": 6, "method": "cg",
         "precision": "df64", "fmt": "sell", "which": 1, "evals": False},
        # A middle-sized 3D grid, steepest descent.
        _fd("fd3d_80_p32_sd", (80, 80, 80), 32, 4, method="sd"),
        # The headline problem: 128^3, p = 64, conjugate gradients.
        _fd("fd3d_128_p64_cg", (128, 128, 128), 64, 4),
        # Dense operators: the mixed-precision form at its full size, and an
        # ordinary one in df64.
        _dense("dense_16k_p128_mixed", 16384, 128, 3, "mixed"),
        _dense("dense_4k_p32_df64", 4096, 32, 6, "df64"),
        # Many uneven graph problems in one graph-captured batch.
        {"name": "batch_48_graphs", "kind": "batch", "nprob": 48, "n_lo": 2048, "n_hi": 65536, "sizes": 4, "steps": 12},
        # The warm-start network: a training step of the small (24 x 24)
        # family, and forward plus subspace loss and its gradient for the
        # wide family (64 operators, coarse 32 x 32, p = 32).
        {"name": "train_24_p4", "kind": "train", "nc": 8, "nf": 24, "p": 4, "hidden": 256, "batch": 64},
        {"name": "warm_loss_64_p32", "kind": "loss", "nc": 32, "nf": 64, "p": 32, "hidden": 512, "batch": 64},
    ]


def _fd(name, dims, p, steps, method="cg", precision="df64", which=1, fmt="csr", evals=False):
    d = list(dims) + [0] * (3 - len(dims))
    c = {"name": name, "kind": "solve", "op": "fd", "d0": d[0], "d1": d[1], "d2": d[2], "p": p, "steps": steps,
         "method": method, "precision": precision, "fmt": fmt, "which": which, "evals": evals}
    if name is None:
        del c["name"]
    return c


def _dense(name, n, p, steps, precision):
    c = {"name": name, "kind": "solve", "op": "dense", "n": n, "p": p, "steps": steps, "method": "cg",
         "precision": precision, "fmt": "csr", "which": 1, "evals": False}
    if name is None:
        del c["name"]
    return c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fd", "fd", "fd", "er", "dense", "batch", "train", "loss"])
    if kind == "fd":
        n = _log_int(rng, 1024, 1_600_000)
        p = _log_int(rng, 4, 64 if n > 100_000 else 100)
        while n < 16 * p:
            p = max(4, p // 2)
        if n < 20_000 and rng.random() < 0.5:
            d0 = max(5, int(math.sqrt(n) * rng.uniform(0.6, 1.5)))
            dims = (d0, max(5, n // d0))
        else:
            s = n ** (1 / 3)
            d0, d1 = (max(5, int(s * rng.uniform(0.7, 1.3))) for _ in range(2))
            dims = (d0, d1, max(5, n // (d0 * d1)))
        f64 = n < 30_000 and rng.random() < 0.2
        return _fd(None, dims, p, rng.randint(3, 8), method=rng.choice(["cg", "cg", "sd"]),
                   precision="f64" if f64 else "df64", which=rng.choice([1, -1]), fmt=rng.choice(["csr", "csr", "sell"]))
    if kind == "er":
        return {"kind": "solve", "op": "er", "n": _log_int(rng, 2048, 120_000), "p": _log_int(rng, 4, 64),
                "steps": rng.randint(3, 8), "method": "cg", "precision": "df64", "fmt": rng.choice(["csr", "sell"]),
                "which": rng.choice([1, -1]), "evals": False}
    if kind == "dense":
        n = _log_int(rng, 512, 8192)
        return _dense(None, n, _log_int(rng, 8, 128 if n >= 2048 else 32), rng.randint(3, 6),
                      rng.choice(["df64", "mixed"]))
    if kind == "batch":
        lo = _log_int(rng, 500, 8000)
        return {"kind": "batch", "nprob": rng.randint(6, 48), "n_lo": lo, "n_hi": lo * rng.randint(2, 8),
                "sizes": rng.randint(0, 1 << 20), "steps": rng.randint(4, 12)}
    nc = rng.randint(6, 32) if kind == "loss" else rng.randint(6, 12)
    return {"kind": kind, "nc": nc, "nf": nc * 2 + rng.randint(1, 8), "p": rng.choice([4, 6, 8, 16, 32 if nc > 8 else 5]),
            "hidden": rng.choice([128, 200, 256, 512]), "batch": rng.randint(8, 64)}


# ---- operators ----------------------------------------------------------------

class _Csr:
    def __init__(self, n, rowptr, colidx, val):
        self.n, self.rowptr, self.colidx, self.val = n, rowptr, colidx, val


def _generator(seed, extra=0):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1000003 + extra)


def _laplacian(dims):
    """Unscaled finite-difference Dirichlet Laplacian (5 or 7 points), columns ascending."""
    n = math.prod(dims)
    idx = torch.arange(n, device=DEV)
    strides, s = [], 1
    for d in dims:
        strides.append(s)
        s *= d
    cols, ok = [], []
    for a in reversed(range(len(dims))):
        cols.append(idx - strides[a])
        ok.append((idx // strides[a]) % dims[a] > 0)
    cols.append(idx)
    ok.append(torch.ones(n, dtype=torch.bool, device=DEV))
    for a in range(len(dims)):
        cols.append(idx + strides[a])
        ok.append((idx // strides[a]) % dims[a] < dims[a] - 1)
    val = torch.full((n, len(cols)), -1.0, dtype=F64, device=DEV)
    val[:, len(dims)] = 2.0 * len(dims)
    cols, ok = torch.stack(cols, 1), torch.stack(ok, 1)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(ok.sum(1), 0)
    return _Csr(n, rowptr, cols[ok].to(torch.int32), val[ok])


def _graph(n, g):
    """Laplacian of a random graph of mean degree about 8 plus a diagonal shift in (0, 1); every entry a float32."""
    u = torch.randint(n, (2, 4 * n), generator=g, device=DEV)
    u = u[:, u[0] != u[1]]
    key = torch.unique(u.min(0).values * n + u.max(0).values)
    lo, hi = key // n, key % n
    shift = torch.rand(n, generator=g, device=DEV, dtype=F64)
    deg = torch.bincount(torch.cat([lo, hi]), minlength=n)
    i = torch.arange(n, device=DEV)
    rows, cols = torch.cat([lo, hi, i]), torch.cat([hi, lo, i])
    val = torch.cat([torch.full((2 * lo.numel(),), -1.0, dtype=F64, device=DEV), (deg + shift).float().double()])
    order = torch.argsort(rows * n + cols)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return _Csr(n, rowptr, cols[order].to(torch.int32), val[order])


def _dense_matrix(n, p, g):
    """Q diag(lam) Q^T, Q a product of 8 Householder reflectors; the top p values a gap of 1e-2 above the rest."""
    i = torch.arange(1, n + 1, device=DEV, dtype=F64)
    lam = 1.0 - i / n
    lam[:p] = 1.0 - (p + 1) / n + 1e-2 + (p - i[:p]) / n
    A = torch.diag(lam)
    for _ in range(8):
        v = torch.randn(n, generator=g, device=DEV, dtype=F64)
        v /= v.norm()
        Av = A @ v
        w = 2.0 * Av - 2.0 * (v @ Av) * v
        A.addr_(v, w, alpha=-1.0)
        A.addr_(w, v, alpha=-1.0)
    return 0.5 * (A + A.T)


def _rows(c):
    return c["n"] if c["op"] != "fd" else math.prod(_dims(c))


def _dims(c):
    return tuple(d for d in (c["d0"], c["d1"], c["d2"]) if d)


def _operator(c, seed):
    if c["op"] == "fd":
        return _laplacian(_dims(c))
    if c["op"] == "er":
        return _graph(c["n"], _generator(seed, 1))
    return gsi.Dense(_dense_matrix(c["n"], c["p"], _generator(seed, 1)))


def _start(n, p, seed, extra=2):
    return torch.randn(n, p, generator=_generator(seed, extra), device=DEV, dtype=F64)


def _batch_sizes(c):
    r = np.random.RandomState(c["sizes"])
    n = r.randint(c["n_lo"], c["n_hi"] + 1, c["nprob"])
    return n, r.choice([4, 8, 16, 32], c["nprob"])


def _batch_parts(c, seed):
    n, p = _batch_sizes(c)
    g = _generator(seed, 1)
    mats = [_graph(int(k), g) for k in n]
    x0 = [_start(int(a), int(b), seed, 100 + i) for i, (a, b) in enumerate(zip(n, p))]
    return n, p, mats, x0


class _BatchInput:
    pass


def _hat(nc, nf):
    """nf x nc linear interpolation from nc interior coarse nodes, zero at the boundary."""
    x = (torch.arange(nf, device=DEV, dtype=F64) + 1) * (nc + 1) / (nf + 1)
    return (1.0 - (x[:, None] - torch.arange(1, nc + 1, device=DEV, dtype=F64)[None, :]).abs()).clamp_min(0.0)


def _network(c, seed):
    """Weights, inputs, S = P^T P (CSR) and Bt = P^T U for smooth orthonormal U."""
    nc, nf, p, h, b = c["nc"], c["nf"], c["p"], c["hidden"], c["batch"]
    g = _generator(seed, 3)
    dout = nc * nc * p
    prm = {}
    for k, (r, q, s) in {"1": (h, 16, 2.0), "2": (h, h, 2.0), "3": (dout, h, 1.0)}.items():
        prm["W" + k] = (torch.randn(r, q, generator=g, device=DEV) * math.sqrt(s / q)).float()
        prm["b" + k] = torch.zeros(r, device=DEV)
    x = torch.randn(b, 16, generator=g, device=DEV)
    P1 = _hat(nc, nf)
    S = torch.kron(P1.T @ P1, P1.T @ P1)
    P = torch.kron(P1, P1)
    U = torch.matmul(P, torch.randn(b, nc * nc, p, generator=g, device=DEV, dtype=F64))
    U = U + 0.1 * torch.randn(b, nf * nf, p, generator=g, device=DEV, dtype=F64)
    Bt = torch.matmul(P.T, torch.linalg.qr(U).Q).float().contiguous()
    keep = S != 0
    rowptr = torch.zeros(nc * nc + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(keep.sum(1), 0)
    col = torch.arange(nc * nc, device=DEV).expand_as(S)[keep].to(torch.int32)
    return prm, x, (rowptr, col.contiguous(), S[keep].contiguous()), Bt, S


# ---- a pass ---------------------------------------------------------------------

def prepare(case, seed):
    c = case
    if c["kind"] == "solve":
        A = _operator(c, seed)
        X0 = _start(A.n, c["p"], seed)
        s = gsi.Solver(A, c["p"], X0, method=c["method"], which=c["which"], precision=c["precision"], fmt=c["fmt"],
                       tol=1e-12)
        return {"case": c, "solver": s, "X0": X0}
    if c["kind"] == "batch":
        n, p, mats, x0 = _batch_parts(c, seed)
        B = _BatchInput()
        nnz = np.array([m.colidx.numel() for m in mats])
        base = np.concatenate([[0], np.cumsum(nnz)])
        B.n, B.p = n, p
        B.rowptr = np.concatenate([[0]] + [m.rowptr[1:].cpu().numpy() + k for m, k in zip(mats, base)])
        B.colidx = torch.cat([m.colidx for m in mats]).cpu().numpy()
        B.val = torch.cat([m.val for m in mats]).float().cpu().numpy()
        x = torch.cat([x.reshape(-1) for x in x0])
        B.X0 = x.cpu().numpy()
        return {"case": c, "batch": gsi.Batch(B, tol=1e-12, max_iters=c["steps"]), "X0": x}
    prm, x, S, Bt, _ = _network(c, seed)
    dout = c["nc"] ** 2 * c["p"]
    net = gsi.MLP(16, c["hidden"], dout, gsi.MLP.flatten({k: v.cpu().numpy() for k, v in prm.items()}),
                  max_batch=c["batch"])
    return {"case": c, "net": net, "x": x, "S": S, "Bt": Bt,
            "out": torch.empty(c["batch"], dout, device=DEV)}


def run(state):
    c = state["case"]
    if c["kind"] == "solve":
        s = state["solver"]
        s.reset(state["X0"])
        s.step(c["steps"])
        if c["precision"] == "mixed":
            # the iterate as the solver holds it: its operator applies carry
            # 21-bit operands, so float64 copies would say nothing more. Copied:
            # the views end with the solver
            return [v.clone() for v in s.state()]
        X, _ = s.basis(evals=False, device=True)
        if not c["evals"]:
            return [X]
        return [X, s.basis(evals=True, device=True)[1]]
    if c["kind"] == "batch":
        b = state["batch"]
        b.restart(state["X0"])
        b.solve(check=False)
        return [b.basis(i, evals=False)[0] for i in range(b.nprob)]
    m, p = c["nc"] ** 2, c["p"]
    if c["kind"] == "train":
        loss = state["net"].train_step(state["x"], state["S"], state["Bt"], m, p, 1e-3)
        return [loss, state["net"].grads()]
    C = state["net"].forward(state["x"], state["out"])
    loss, dC = gsi.warm_loss_grad(C.view(c["batch"], m, p), state["S"], state["Bt"], m, p, gscale=1.0 / c["batch"])
    return [C, loss.float(), dC]  # float32 as the network's other outputs


def work(case):
    """Per iteration: the operator once, 15 block reads or writes (X, Y, R, the
    last R, P, D and W, each product's operands once) and nine n x p x p
    products; the start two polar steps and an apply."""
    c = case
    if c["kind"] == "solve":
        return _work_solve(c, _rows(c), c["p"], c["steps"])
    if c["kind"] == "batch":
        n, p = _batch_sizes(c)
        tot = {"bytes": 0.0, "flops": 0.0}
        for a, b in zip(n, p):
            w = _work_solve({"op": "er32", "precision": "df64", "method": "cg"}, int(a), int(b), c["steps"])
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    m, p, b, h = c["nc"] ** 2, c["p"], c["batch"], c["hidden"]
    params = h * 16 + h * h + m * p * h
    back = c["kind"] == "train"
    return {"bytes": 4.0 * params * (9 if back else 1) + 4.0 * b * m * p * 3,
            "flops": 2.0 * b * params * (3 if back else 1) + 2.0 * b * m * p * p * 4}


def _work_solve(c, n, p, steps):
    nnz = {"fd": 7.0 if c.get("d2") else 5.0, "er": 9.0, "er32": 9.0, "dense": float(n)}[c["op"]] * n
    entry = {"dense": 8.0, "er32": 8.0}.get(c["op"], 12.0)
    cg = c["method"] == "cg"
    applies = steps + 1
    blocks = steps * (15 if cg else 11) + 8
    products = steps * (9 if cg else 7) + 4
    return {"bytes": applies * entry * nnz + blocks * 8.0 * n * p,
            "flops": applies * 2.0 * nnz * p + products * 2.0 * n * p * p}


# ---- the same in 64 bits, with torch and numpy alone ----------------------------

def _sym(M):
    return 0.5 * (M + M.T)


def _inv_sqrt(S):
    w, V = torch.linalg.eigh(S)
    return (V / w.sqrt()) @ V.T


def _step_length(al, be, ga, ze):
    """The first minimiser of the trace model past the smallest branch root."""
    def slope(t):
        return -np.sum((ze + (ga - al * be) * t - be * ze * t * t) / (1.0 + be * t * t) ** 2)

    use = (be > 2.220446049250313e-16 * be.sum()) & (ze > 0)
    if not use.any():
        return 0.0
    b, z = be[use], ze[use]
    d = ga[use] - al[use] * b
    disc = np.sqrt(d * d + 4.0 * b * z * z)
    xi = np.where(d < 0, 2.0 * z / (disc - d + (d >= 0)), (d + disc) / (2.0 * b * z))
    lo, hi = 0.0, xi.min()
    k = 0
    while slope(hi) < 0 and k < 64:
        lo, hi, k = hi, min(2.0 * hi, xi.max()) if hi < xi.max() else 2.0 * hi, k + 1
    for _ in range(120):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if slope(mid) < 0 else (lo, mid)
    return 0.5 * (lo + hi)


def _iterate(apply, X0, steps, cg):
    X = X0
    for _ in range(2):
        X = X @ _inv_sqrt(_sym(X.T @ X))
    P = Rp = None
    rr_prev = 0.0
    for _ in range(steps):
        Y = apply(X)
        C = _sym(X.T @ Y)
        R = Y - X @ C
        rr = float((R * R).sum())
        D = R
        if cg and P is not None:
            b = (rr - float((R * Rp).sum())) / rr_prev
            D = R + b * (P - X @ (X.T @ P))
            if float((D * R).sum()) <= 0:
                D = R
        W = apply(D)
        B = _sym(D.T @ D)
        be, V = torch.linalg.eigh(B)
        be = be.clamp_min(0.0)

        def diag(M):
            return (V * (M @ V)).sum(0).cpu().numpy()

        t = _step_length(diag(C), be.cpu().numpy(), diag(_sym(D.T @ W)), diag(D.T @ R))
        Z = X + t * D
        X = Z @ _inv_sqrt(_sym(Z.T @ Z))
        P, Rp, rr_prev = D, R, rr
    return X


def _apply_of(A, which):
    if isinstance(A, gsi.Dense):
        return lambda V: which * (A.val @ V)
    M = torch.sparse_csr_tensor(A.rowptr, A.colidx.long(), A.val * which, (A.n, A.n))
    return lambda V: M @ V


def exact(case, seed):
    c = case
    if c["kind"] == "solve":
        A = _operator(c, seed)
        apply = _apply_of(A, c["which"])
        X = _iterate(apply, _start(A.n, c["p"], seed), c["steps"], c["method"] == "cg")
        if c["precision"] == "mixed":
            return [_pairs(X), _pairs(apply(X))]
        if not c["evals"]:
            return [X]
        return [X, c["which"] * torch.linalg.eigvalsh(_sym(X.T @ apply(X))).flip(0)]
    if c["kind"] == "batch":
        out = []
        for A, x0 in zip(*_batch_parts(c, seed)[2:]):
            out.append(_iterate(_apply_of(A, 1), x0, c["steps"], True))
        return out
    prm, x, _, Bt, S = _network(c, seed)
    b, m, p = c["batch"], c["nc"] ** 2, c["p"]

    def bf(t):  # operands of the network's products are bfloat16 by contract
        return t.float().bfloat16().double()

    w = {k: v.double() for k, v in prm.items()}
    h1 = (bf(x) @ bf(w["W1"]).T + w["b1"]).clamp_min(0.0)
    h2 = (bf(h1) @ bf(w["W2"]).T + w["b2"]).clamp_min(0.0)
    C = bf(h2) @ bf(w["W3"]).T + w["b3"]
    Cs, Bd = C.view(b, m, p), Bt.double()
    SC = torch.matmul(S, Cs)
    N, G = Cs.mT @ SC, Bd.mT @ Cs
    Ni = torch.linalg.inv(0.5 * (N + N.mT))
    Q = G.mT @ G
    loss = p - (Ni @ Q).diagonal(dim1=1, dim2=2).sum(1)
    dC = (-2.0 / b) * (Bd @ (G @ Ni) - SC @ (Ni @ Q @ Ni))
    if c["kind"] == "loss":
        return [C, loss, dC]
    d3 = dC.reshape(b, m * p)
    d2 = (bf(d3) @ bf(w["W3"])) * (h2 > 0)
    d1 = (bf(d2) @ bf(w["W2"])) * (h1 > 0)
    return [loss.mean().reshape(()),
            {"W1": bf(d1).T @ bf(x), "b1": d1.sum(0), "W2": bf(d2).T @ bf(h1), "b2": d2.sum(0),
             "W3": bf(d3).T @ bf(h2), "b3": d3.sum(0)}]


def _pairs(X):
    hi = X.float()
    return torch.stack([hi, (X - hi.double()).float()], -1)
