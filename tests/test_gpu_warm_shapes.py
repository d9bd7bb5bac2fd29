"""The warm-start kernels where their tiles end: bf16 products in every staging
of the operands (along k, along i, element by element) and both tile sizes,
and the subspace loss for rows and widths that fill no block."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["nt", "nn", "tn", "strided", "offset"])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (33, 31, 17), (64, 96, 32), (65, 130, 100), (64, 300, 257),
                                   (700, 1100, 45)])
def test_gemm_bf16_layouts(torch_cuda, M, N, K, layout):
    torch = torch_cuda
    from paper_2306_10379_gb300 import gsi
    g = torch.Generator(device="cuda").manual_seed(M + N + K)

    def rand(*s):
        return torch.randn(*s, generator=g, device="cuda")

    if layout == "nt":      # A[i][k], B[j][k]
        a, b = rand(M, K), rand(N, K)
        A, sa, Am, B, sb, Bm = a, (K, 1), a, b, (1, K), b.T
    elif layout == "nn":    # A[i][k], B[k][j]
        a, b = rand(M, K), rand(K, N)
        A, sa, Am, B, sb, Bm = a, (K, 1), a, b, (N, 1), b
    elif layout == "tn":    # A[k][i], B[k][j]
        a, b = rand(K, M), rand(K, N)
        A, sa, Am, B, sb, Bm = a, (1, M), a.T, b, (N, 1), b
    elif layout == "strided":  # neither index contiguous
        a, b = rand(M, K, 3), rand(K, N, 2)
        A, sa, Am, B, sb, Bm = a, (3 * K, 3), a[..., 0], b, (2 * N, 2), b[..., 0]
    else:                   # rows off 16 bytes
        a, b = rand(M * K + 1)[1:].view(M, K), rand(N * K + 3)[3:].view(N, K)
        A, sa, Am, B, sb, Bm = a, (K, 1), a, b, (1, K), b.T
    bias, mask = rand(N), rand(M, N)
    C = rand(M, N)
    C0 = C.clone()
    gsi.gemm_bf16(M, N, K, A, sa, B, sb, C, N, alpha=0.5, beta=2.0, bias=bias, mask=mask, relu=True)
    x, y = Am.bfloat16().double(), Bm.bfloat16().double()
    ref = 0.5 * (x @ y) + 2.0 * C0.double() + bias.double()
    size = 0.5 * (x.abs() @ y.abs()) + 2.0 * C0.double().abs() + bias.double().abs()
    ref = torch.where(mask > 0, ref, torch.zeros_like(ref)).clamp_min(0.0)
    # K float32 additions of exact products, then three more roundings
    assert bool(((C.double() - ref).abs() <= (K + 4) * 2.0 ** -24 * size).all())


@pytest.mark.parametrize("m,p,batch", [(1, 1, 1), (9, 2, 3), (31, 5, 2), (128, 7, 2), (129, 33, 3), (300, 64, 2)])
def test_loss_and_gradient_shapes(torch_cuda, m, p, batch):
    torch = torch_cuda
    from paper_2306_10379_gb300 import gsi
    rng = np.random.default_rng(m * 100 + p)
    # a symmetric positive definite S with rows of uneven length, the longest
    # ones together beyond what a block stages
    S = np.where(rng.random((m, m)) < 0.15, rng.uniform(-0.1, 0.1, (m, m)), 0.0)
    S = S + S.T
    S[np.arange(m), np.arange(m)] = 1.0 + np.abs(S).sum(1)
    rows, cols = np.nonzero(S)
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=m))])
    csr = tuple(torch.as_tensor(v, device="cuda") for v in
                (rp.astype(np.int64), cols.astype(np.int32), S[rows, cols].astype(np.float64)))
    C = rng.standard_normal((batch, m, p)).astype(np.float32)
    Bt = (rng.standard_normal((batch, m, p)) / np.sqrt(m)).astype(np.float32)
    loss, dC = gsi.warm_loss_grad(torch.as_tensor(C, device="cuda"), csr, torch.as_tensor(Bt, device="cuda"), m, p,
                                  gscale=0.5)
    for s in range(batch):
        c, b = C[s].astype(np.float64), Bt[s].astype(np.float64)
        N, G = c.T @ S @ c, b.T @ c
        Ni = np.linalg.inv(0.5 * (N + N.T))
        Q = G.T @ G
        ref = p - np.trace(Ni @ Q)
        d = -2.0 * 0.5 * (b @ (G @ Ni) - S @ c @ (Ni @ Q @ Ni))
        # N and G carry float32 sums of 32 terms; their errors pass through N^{-1}
        eps = 40 * 2.0 ** -24 * np.linalg.cond(N)
        assert abs(float(loss[s]) - ref) <= eps * p
        assert np.linalg.norm(dC[s].cpu().numpy() - d) <= eps * max(np.linalg.norm(b) * np.linalg.norm(G @ Ni),
                                                                   np.linalg.norm(d))
