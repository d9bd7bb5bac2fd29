"""The df64 p x p step at the edges of its block shapes (p = 16, 32, 64 and
their neighbours, odd p, the largest) and for spectra of B = D^T D that the
float32 sweeps cannot resolve alone: graded over 12 decades, clustered,
rank-deficient and zero."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _inv_sqrt(S):
    w, V = np.linalg.eigh(S)
    return (V / np.sqrt(w)) @ V.T


def _problem(p, kind, rng):
    n = 4 * p + 9
    Q, _ = np.linalg.qr(rng.standard_normal((n, p)))
    A = rng.standard_normal((n, n))
    A = A + A.T
    C = Q.T @ A @ Q
    C = 0.5 * (C + C.T)
    R = A @ Q - Q @ C
    U, _ = np.linalg.qr(rng.standard_normal((p, p)))
    tau = {"plain": np.ones(p), "graded": 10.0 ** -np.linspace(0, 6, p),
           "clustered": np.where(np.arange(p) < p // 2, 1.0, 1.0 + 1e-9 * np.arange(p)),
           "rank": np.where(np.arange(p) < max(1, p // 3), 1.0, 0.0), "zero": np.zeros(p)}[kind]
    if kind == "clustered":  # B itself clustered, not only the scaling
        w, V = np.linalg.eigh(R.T @ R)
        R0 = R @ (V / np.sqrt(w)) @ U
        D = R0 * tau
        D = D @ np.linalg.qr(rng.standard_normal((p, p)))[0]
    else:
        D = R @ (U * tau) @ U.T
    return Q, A, C, R, D


def _phi_slope(t, C, B, Gam, Z):
    """phi'(t) of phi(t) = -1/2 tr((C + t (Z + Z^T) + t^2 Gam)(I + t^2 B)^-1), and the size of its terms."""
    I = np.eye(B.shape[0])
    S = np.linalg.inv(I + t * t * B)
    N = C + t * (Z + Z.T) + t * t * Gam
    a = np.trace((Z + Z.T + 2 * t * Gam) @ S)
    b = np.trace(N @ S @ (2 * t * B) @ S)
    return -0.5 * (a - b), 0.5 * (np.abs((Z + Z.T + 2 * t * Gam) * S.T).sum() + np.abs(N * (S @ (2 * t * B) @ S).T).sum())


@pytest.mark.parametrize("kind", ["plain", "graded", "clustered", "rank", "zero"])
@pytest.mark.parametrize("p", [1, 2, 7, 8, 15, 16, 17, 31, 32, 33, 48, 63, 64, 65, 97, 127, 128])
def test_step_and_polar_factor(torch_cuda, p, kind):
    torch = torch_cuda
    from paper_2306_10379_gb300 import gsi
    rng = np.random.default_rng(100 * p + len(kind))
    X, A, C, R, D = _problem(p, kind, rng)
    W = A @ D
    B, Gam, Z, XX, XD = D.T @ D, D.T @ W, D.T @ R, X.T @ X, X.T @ D
    Gam = 0.5 * (Gam + Gam.T)

    def dev(m):
        return torch.as_tensor(np.ascontiguousarray(m), device="cuda")

    M = torch.empty((p, p), dtype=torch.float64, device="cuda")
    out = torch.zeros(16, dtype=torch.float64, device="cuda")
    gsi.linesearch(*(dev(m) for m in (C, B, Gam, Z, XX, XD)), M, out)
    o = out.cpu().numpy()
    assert o[3] == 0.0
    t = float(o[0])
    if kind == "zero":
        assert t == 0.0
    elif t == 0.0:
        # no branch descends: zeta = diag(V^T Z V) <= 0 in the eigenbasis, so
        # its sum, the trace of Z, is not positive either
        assert kind == "clustered" and np.trace(Z) <= 0.0
    else:
        # the coefficients carry p df64 products (2^-46 of their terms each),
        # so phi' vanishes to p 2^-45 of the sum of its terms
        slope, size = _phi_slope(t, C, B, Gam, Z)
        assert t > 0.0 and abs(slope) <= p * 2.0 ** -45 * size
    S = XX + t * (XD + XD.T) + t * t * B
    S = 0.5 * (S + S.T)
    Mr = _inv_sqrt(S)
    w = np.linalg.eigvalsh(S)
    # the products perturb S by at most p 2^-45 ||S||, and S^{-1/2} by that
    # over 2 s_min^{3/2}; M itself is two more such products
    bound = max(4, p) * 2.0 ** -45 * (np.linalg.norm(Mr) + np.sqrt(p) * w[-1] / w[0] ** 1.5)
    assert np.linalg.norm(M.cpu().numpy() - Mr) <= bound
    assert abs(o[4] - np.linalg.eigvalsh(B)[-1]) <= max(4, p) * 2.0 ** -45 * max(o[4], 1e-300)
