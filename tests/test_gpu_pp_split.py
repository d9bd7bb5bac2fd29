"""The df64 p x p step in the two launches of the solver: both forms of the
eigenbasis for 32 < p <= 64 (one CTA, which large n takes, and a cluster),
spectra of B whose gaps put the corrections K on either side of their limits,
and the next K = M (X^T D + t B), which is a float64 product."""
import numpy as np
import pytest

from oracle import gsi_oracle as O
from paper_2306_10379_gb300 import inputs as I
from tests.test_gpu_pp_step import _inv_sqrt, _phi_slope, _problem

pytestmark = pytest.mark.gpu


def _step(torch, C, B, Gam, Z, XX, K, beta, cluster):
    from paper_2306_10379_gb300 import gsi
    p = B.shape[0]

    def dev(m):
        return torch.as_tensor(np.ascontiguousarray(m), device="cuda")

    M, Kn = (torch.empty((p, p), dtype=torch.float64, device="cuda") for _ in range(2))
    out = torch.zeros(16, dtype=torch.float64, device="cuda")
    gsi.pp_step(*(dev(m) for m in (C, B, Gam, Z, XX, K)), beta, M, Kn, out, cluster=cluster)
    return M.cpu().numpy(), Kn.cpu().numpy(), out.cpu().numpy()


def _grams(X, A, D, R):
    W = A @ D
    Gam = D.T @ W
    return D.T @ D, 0.5 * (Gam + Gam.T), D.T @ R, X.T @ X


def _check_polar(M, S, p):
    # the bound of test_gpu_pp_step: p 2^-45 ||S|| in S, two more products
    w = np.linalg.eigvalsh(S)
    Mr = _inv_sqrt(S)
    assert np.linalg.norm(M - Mr) <= max(4, p) * 2.0 ** -45 * (np.linalg.norm(Mr) + np.sqrt(p) * w[-1] / w[0] ** 1.5)


@pytest.mark.parametrize("cluster", [False, True])
@pytest.mark.parametrize("kind", ["plain", "graded", "clustered", "rank", "zero"])
@pytest.mark.parametrize("p", [33, 48, 63, 64])
def test_both_forms_of_the_eigenbasis(torch_cuda, p, kind, cluster):
    rng = np.random.default_rng(100 * p + len(kind))
    X, A, C, R, D = _problem(p, kind, rng)
    B, Gam, Z, XX = _grams(X, A, D, R)
    M, _, o = _step(torch_cuda, C, B, Gam, Z, XX, np.zeros((p, p)), 0.0, cluster)
    assert o[3] == 0.0
    t = float(o[0])
    if kind == "zero":
        assert t == 0.0
    elif t == 0.0:
        assert kind == "clustered" and np.trace(Z) <= 0.0
    else:
        slope, size = _phi_slope(t, C, B, Gam, Z)
        assert t > 0.0 and abs(slope) <= p * 2.0 ** -45 * size
    XD = (np.eye(p) - XX) @ C
    S = XX + t * (XD + XD.T) + t * t * B
    _check_polar(M, 0.5 * (S + S.T), p)


@pytest.mark.parametrize("lo", [-8, -7, -6, -5, -4, -3, -2, -1])
@pytest.mark.parametrize("p,cluster", [(8, False), (16, False), (32, False), (48, False), (48, True), (128, True)])
def test_gaps_around_the_limits(torch_cuda, p, cluster, lo):
    """Gaps of B between 10^lo and 10^(lo + 1) of its norm: after the float32
    sweeps F is about 10^-7, so that K crosses its limits over these rows."""
    rng = np.random.default_rng(10 * p - lo)
    X, A, C, R, _ = _problem(p, "plain", rng)
    n = X.shape[0]
    Q = np.linalg.qr(np.hstack([X, rng.standard_normal((n, p))]))[0][:, p:]
    w = 1.0 + np.cumsum(10.0 ** rng.uniform(lo, lo + 1, p)) / p
    D = (Q * np.sqrt(w)) @ np.linalg.qr(rng.standard_normal((p, p)))[0].T
    B, Gam, _, XX = _grams(X, A, D, R)
    Z = B  # a descent direction: every zeta positive
    M, _, o = _step(torch_cuda, C, B, Gam, Z, XX, np.zeros((p, p)), 0.0, cluster)
    t = float(o[0])
    assert o[3] == 0.0 and t > 0.0
    XD = (np.eye(p) - XX) @ C
    S = XX + t * (XD + XD.T) + t * t * B
    _check_polar(M, 0.5 * (S + S.T), p)


@pytest.mark.parametrize("p,cluster", [(1, False), (4, False), (8, False), (15, False), (16, False), (17, False),
                                       (32, False), (33, False), (64, False), (64, True), (65, True), (128, True)])
def test_next_k_is_a_float64_product(torch_cuda, p, cluster):
    rng = np.random.default_rng(p)
    X, A, C, R, D = _problem(p, "plain", rng)
    B, Gam, Z, XX = _grams(X, A, D, R)
    K = 1e-3 * rng.standard_normal((p, p))
    beta = 0.7
    M, Kn, o = _step(torch_cuda, C, B, Gam, Z, XX, K, beta, cluster)
    L = np.longdouble
    E = np.eye(p, dtype=L) - 0.5 * (XX + XX.T).astype(L)
    XD = E @ (C.astype(L) + L(beta) * K.astype(L))
    T = XD + L(o[0]) * (0.5 * (B + B.T)).astype(L)
    ref = M.astype(L) @ T
    # p float64 additions; X^T D = (I - XX)(C + beta K) carries df64 rounding
    # of the (rounding-level) I - XX
    size = np.abs(M) @ np.abs(T).astype(np.float64)
    xd = np.abs(M) @ (np.abs(E).astype(np.float64) @ (np.abs(C) + beta * np.abs(K)))
    assert np.all(np.abs(Kn - ref) <= (p + 3) * 2.0 ** -53 * size + (p + 4) * 2.0 ** -45 * xd)


@pytest.mark.parametrize("p", [33, 64])
def test_large_n_solver_steps(torch_cuda, p):
    """n >= 250,000 and 32 < p <= 64: the eigenbasis on one CTA, in the solver."""
    from paper_2306_10379_gb300 import gsi
    A = I.fd_laplacian((64, 64, 62))
    assert A.n >= 250000
    X0 = np.random.default_rng(p).standard_normal((A.n, p))
    ref = []
    O.solve(O.csr_operator(A.n, A.rowptr, A.colidx, A.val), X0, O.Options(method="cg", tol=1e-12, max_iters=2),
            callback=lambda k, X, Y, t: ref.append((X.copy(), t)))
    with gsi.Solver(A, p, X0, method="cg", tol=1e-12) as s:
        for Xr, tr in ref:
            t = s.step(1)["last_step"]
            X, _ = s.basis(evals=False)
            assert abs(t - tr) <= 1e-10 * abs(tr)
            assert np.max(np.abs(X - Xr)) <= 1e-10
