"""The batched solver's line-search Grams on an operator that is symmetric only
up to a perturbation: D^T W enters as the average with its transpose, as in
the single-problem solver and the oracle."""
import numpy as np
import pytest

from oracle import gsi_oracle as O
from paper_2306_10379_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [2, 4, 8, 16, 32])
def test_unsymmetric_operator(torch_cuda, p):
    from paper_2306_10379_gb300 import gsi
    n = np.array([2 * p + r for r in (9, 65, 257, 513)], np.int32)
    B = I.er_batch(4, I.SEED_BASE + 80 + p, sizes=(n, np.full(4, p, np.int32)))
    rng = np.random.default_rng(p)
    B.val = (B.val * (1.0 + 0.05 * rng.standard_normal(B.val.size))).astype(np.float32)
    mats, k = [], 0
    for m in B.mats:
        nnz = len(m.val)
        mats.append(O.csr_operator(m.n, m.rowptr, m.colidx, B.val[k:k + nnz]))
        k += nnz
    an = np.array([O.anorm_inf(A) for A in mats])
    K = 3
    ref = [[] for _ in mats]
    # plain gradients: with A unsymmetric X^T D of the CG closed form differs by the skew part of C
    O.batched_solve(mats, B.X0s, O.Options(method="sd", tol=1e-12, max_iters=K), anorms=an,
                    callback=lambda i, k, X, Y, t: ref[i].append((X.copy(), t)))
    with gsi.Batch(B, method="sd", tol=1e-12, anorm=an) as b:
        for k in range(K):
            b.step(1)
            for i in range(4):
                X, _ = b.basis(i, evals=False)
                Xr, tr = ref[i][k]
                assert abs(b.info(i)["last_step"] - tr) <= 1e-10 * abs(tr), (i, k)
                assert np.max(np.abs(X - Xr)) <= 1e-10, (i, k)
