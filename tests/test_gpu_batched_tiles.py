"""The batched solver's tile kernels at the edges of their chunks: every block
width, row counts around the staged chunks (8 to 256 rows in the Gram kernel,
64 to 512 in the row kernels) and operators scaled by powers of two, against
the oracle's iterates."""
import numpy as np
import pytest

from oracle import gsi_oracle as O
from paper_2306_10379_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ROWS = (7, 8, 9, 63, 65, 129, 255, 257, 513)


@pytest.mark.parametrize("p", [2, 4, 8, 16, 32])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 20, 2.0 ** -20])
def test_tile_edges(torch_cuda, p, scale):
    from paper_2306_10379_gb300 import gsi
    n = np.array([2 * p + r for r in ROWS], np.int32)
    B = I.er_batch(len(ROWS), I.SEED_BASE + 40 + p, sizes=(n, np.full(len(ROWS), p, np.int32)))
    B.val = (B.val * np.float32(scale)).astype(np.float32)
    mats = [O.csr_operator(m.n, m.rowptr, m.colidx, (m.val * np.float32(scale)).astype(np.float32))
            for m in B.mats]
    an = np.array([O.anorm_inf(A) for A in mats])
    K = 3
    ref = [[] for _ in mats]
    O.batched_solve(mats, B.X0s, O.Options(method="cg", tol=1e-12, max_iters=K), anorms=an,
                    callback=lambda i, k, X, Y, t: ref[i].append((X.copy(), t)))
    with gsi.Batch(B, method="cg", tol=1e-12, anorm=an) as b:
        for k in range(K):
            b.step(1)
            for i in range(len(ROWS)):
                X, _ = b.basis(i, evals=False)
                Xr, tr = ref[i][k]
                assert abs(b.info(i)["last_step"] - tr) <= 1e-10 * abs(tr), (i, k)
                assert np.max(np.abs(X - Xr)) <= 1e-10, (i, k)
                # the measured Gram matrix carries at most about 2^-45 of its
                # norm, the polar factor and the row products 2^-46 sqrt(p)
                assert np.max(np.abs(X.T @ X - np.eye(p))) <= 2e-13, (i, k)
