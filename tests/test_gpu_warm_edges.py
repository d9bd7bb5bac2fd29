"""The warm-start network where a call can go wrong without a wrong size: a
captured training step that outlives a larger one, and samples whose data or
whose N are bad, and operators far from one in scale."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _mass(torch, nc):
    """P^T P of the bilinear prolongation is close to this tensor product (CSR, CUDA)."""
    T = np.diag(np.full(nc, 2.0 / 3.0)) + np.diag(np.full(nc - 1, 1.0 / 6.0), 1) + np.diag(np.full(nc - 1, 1.0 / 6.0), -1)
    S = np.kron(T, T)
    r, c = np.nonzero(S)
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=nc * nc))])
    return S, tuple(torch.as_tensor(v, device="cuda")
                    for v in (rp.astype(np.int64), c.astype(np.int32), S[r, c].astype(np.float64)))


def test_captured_step_after_a_larger_one(torch_cuda):
    """Warm-up, a captured step, a larger eager step, then a replay: the
    replay's gradients are those of an eager step from the same weights."""
    import ctypes
    torch = torch_cuda
    from paper_2306_10379_gb300 import gsi
    nc, p, hid, big, small = 6, 4, 64, 48, 3
    m = nc * nc
    S, csr = _mass(torch, nc)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(big, 16, generator=g, device="cuda")
    Bt = torch.randn(big, m, p, generator=g, device="cuda") / m
    w0 = 0.2 * np.random.default_rng(5).standard_normal(gsi.mlp_num_params(16, hid, m * p)).astype(np.float32)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    net = gsi.MLP(16, hid, m * p, w0, max_batch=big, stream=st)
    xs, bs = x[:small].contiguous(), Bt[:small].contiguous()
    st.wait_stream(torch.cuda.current_stream())

    def enqueue():
        f = gsi._f32
        s = gsi.lib().gsi_warm_train_step(net._ctx, small, f(xs), m, p, gsi._dptr(csr[0], torch.int64),
                                          gsi._dptr(csr[1], torch.int32), gsi._dptr(csr[2], torch.float64), f(bs),
                                          ctypes.c_double(1e-3), None)
        assert s == gsi.GSI_OK

    with torch.cuda.stream(st):
        net.train_step(xs, csr, bs, m, p, 1e-3)
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        enqueue()
        graph.capture_end()
        net.train_step(x, csr, Bt, m, p, 1e-3)  # needs a larger scratch
        for _ in range(3):
            prm = gsi.MLP.flatten(net.params())
            graph.replay()
            st.synchronize()
            got = net.grads()
            ref_net = gsi.MLP(16, hid, m * p, prm, max_batch=big, stream=st)
            ref_net.train_step(xs, csr, bs, m, p, 1e-3)
            ref = ref_net.grads()
            for k in ref:
                assert np.all(np.isfinite(got[k])) and np.array_equal(got[k], ref[k]), k
            net.train_step(x, csr, Bt, m, p, 1e-3)
    del graph


@pytest.mark.parametrize("what", ["nan", "inf"])
def test_bad_samples(torch_cuda, what):
    """dC = 0 only where N is not positive definite: NaN or infinity in a
    sample's Bt shows in its loss and gradient; the other samples are as without it."""
    torch = torch_cuda
    from paper_2306_10379_gb300 import gsi
    nc, p, batch = 5, 4, 4
    m = nc * nc
    S, csr = _mass(torch, nc)
    g = torch.Generator(device="cuda").manual_seed(6)
    C = torch.randn(batch, m, p, generator=g, device="cuda")
    Bt = torch.randn(batch, m, p, generator=g, device="cuda") / m
    C[3, :, 1] = 0.0  # N singular
    loss0, dC0 = gsi.warm_loss_grad(C, csr, Bt, m, p)
    Bt[1, 7, 2] = float(what)
    loss, dC = gsi.warm_loss_grad(C, csr, Bt, m, p)
    for s in (0, 2):
        assert torch.equal(loss[s], loss0[s]) and torch.equal(dC[s], dC0[s]) and bool(torch.isfinite(dC[s]).all())
    assert not bool(torch.isfinite(loss[1]))
    # G = Bt^T C is not finite in a whole row, so no row of dC can be
    assert not bool(torch.isfinite(dC[1]).any())
    for q in (loss0, loss):
        assert bool(torch.isnan(q[3]))
    assert bool((dC0[3] == 0).all()) and bool((dC[3] == 0).all())


@pytest.mark.parametrize("scale", [1.0, 1e-42, 1e42, 1e-150])
def test_scaled_operator(torch_cuda, scale):
    """S of any float64 scale: N = C^T S C in range, loss and dC C^T unchanged
    by S -> a S, C -> C / sqrt(a) (a power of two), Bt as it is scaled."""
    torch = torch_cuda
    from paper_2306_10379_gb300 import gsi
    nc, p, batch = 7, 5, 3
    m = nc * nc
    a = 2.0 ** (2 * round(np.log2(scale) / 2))
    c = 2.0 ** np.clip(round(np.log2(1.0 / a) / 2), -60, 60)  # C stays a float32, and C^T S C too
    rng = np.random.default_rng(8)
    S, csr = _mass(torch, nc)
    S = S * (1.0 + 0.1 * rng.random(S.shape))  # 53-bit values
    S = 0.5 * (S + S.T)
    r, col = np.nonzero(S)
    sv = torch.as_tensor(a * S[r, col], device="cuda")
    C = (c * rng.standard_normal((batch, m, p))).astype(np.float32)
    Bt = (rng.standard_normal((batch, m, p)) / (m * c)).astype(np.float32)
    loss, dC = gsi.warm_loss_grad(torch.as_tensor(C, device="cuda"), (csr[0], csr[1], sv),
                                  torch.as_tensor(Bt, device="cuda"), m, p)
    for s in range(batch):
        c64, b64 = C[s].astype(np.float64), Bt[s].astype(np.float64)
        SC = (a * S) @ c64
        if np.abs(SC).max() < 1e-30:  # S C underflows in float32: N is zero, not positive definite
            assert np.isnan(float(loss[s])) and bool((dC[s] == 0).all())
            continue
        N, G = c64.T @ SC, b64.T @ c64
        Ni = np.linalg.inv(0.5 * (N + N.T))
        Q = G.T @ G
        # as test_gpu_warm_shapes: N and G carry float32 sums of 32 terms
        eps = 40 * 2.0 ** -24 * np.linalg.cond(N)
        tr = np.trace(Ni @ Q)
        assert abs(float(loss[s]) - (p - tr)) <= eps * max(p, tr)
        d = -2.0 * (b64 @ (G @ Ni) - SC @ (Ni @ Q @ Ni))
        assert np.linalg.norm(dC[s].cpu().numpy() - d) <= eps * max(np.linalg.norm(b64) * np.linalg.norm(G @ Ni),
                                                                   np.linalg.norm(d))
