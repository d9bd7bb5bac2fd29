"""The dense digit apply where its tiles end: sizes around 128 rows, 32-row
sub-chunks and the exponent chunks (64, 160, 384 rows), widths around the 32,
64 and 128 columns of a CTA, and A not symmetric (the apply is A^T X)."""
import numpy as np
import pytest

from paper_2306_10379_gb300 import gsi as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nd", [7, 3])
@pytest.mark.parametrize("n,p", [(1, 1), (31, 2), (32, 32), (33, 33), (127, 64), (128, 65), (129, 31), (160, 128),
                                 (161, 17), (384, 64), (386, 96), (770, 127), (1030, 66)])
def test_dense_apply_shapes(torch_cuda, n, p, nd):
    torch = torch_cuda
    rng = np.random.default_rng(1000 * n + p)
    A = G.from_df(G.to_df(rng.standard_normal((n, n)) * 10.0 ** rng.uniform(-3, 3, n)))
    X = G.from_df(G.to_df(rng.standard_normal((n, p))))
    W = torch.full((n, p, 2), float("nan"), device="cuda")
    G.oz_dense_apply(torch.from_numpy(G.to_df(A)).cuda(), torch.from_numpy(G.to_df(X)).cuda(), W, nd=nd)
    got = G.from_df(W.cpu().numpy())
    ref = A.T @ X
    # products cut at the column maxima of an exponent chunk: 2^-44 (7 digits)
    # or 2^-19 (3) of their product per row
    ec = 160 if nd == 7 else (384 if n % 2 == 0 and p % 2 == 0 else 64)
    bound = np.zeros_like(ref)
    for r0 in range(0, n, ec):
        bound += np.outer(np.abs(A[r0:r0 + ec]).max(0), np.abs(X[r0:r0 + ec]).max(0)) * min(ec, n - r0)
    scale = 2.0 ** -44 if nd == 7 else 2.0 ** -19
    assert np.all(np.abs(got - ref) <= scale * bound + 2.0 ** -46 * (np.abs(A.T) @ np.abs(X)))
