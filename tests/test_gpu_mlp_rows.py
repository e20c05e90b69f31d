"""The row-tile training kernels at the edges of their tiles and grids, against the FP64
reference network (oracle/mlp_ref.py): single rows, tile sizes and their neighbours, the change
of tile size of the FP32 kernel (2432 / 2433 rows), more tiles than CTAs, unaligned inputs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp_ref as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2504_20742_gb300 as P
    return P


def _data(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, 16)).astype(np.float32)
    Y = rng.standard_normal((n, 10)).astype(np.float32)
    M = (rng.uniform(size=(n, 10)) > 0.25).astype(np.float32)
    return X, Y, M


def _params():
    theta = R.init_params(3).astype(np.float32)
    return theta + (0.01 * np.random.default_rng(5).standard_normal(theta.size)).astype(np.float32)


# FP32: products of 128 terms and batch sums in FP32 (1e-4, as the gradient test of 64 rows);
# tensor cores: operands rounded to BF16 (2^-9 each), independent over the batch: 1e-2 of the
# gradient's norm, 5e-2 for a single row, whose roundings do not average.
@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 127, 129, 2432, 2433, 20011])
@pytest.mark.parametrize("tc", [False, True])
def test_gradient_at_tile_edges(P, n, tc):
    theta = _params()
    X, Y, M = _data(n, 11 + n)
    Lr, gr = R.loss_and_grad(theta.astype(np.float64), X.astype(np.float64), Y.astype(np.float64), M.astype(np.float64))
    d = "cuda"
    # a batch that starts 4 bytes off a 16-byte boundary takes the scalar copies
    for off in (0, 1):
        buf = torch.zeros(n * 16 + 1, device=d)
        Xt = buf[off:off + n * 16].view(n, 16)
        Xt.copy_(torch.tensor(X))
        p = torch.zeros(theta.size + 1, device=d)[off:off + theta.size]
        p.copy_(torch.tensor(theta))
        Yt, Mt = torch.tensor(Y, device=d), torch.tensor(M, device=d)
        wb = P.ct_mlp_work_bytes(n)
        work = torch.full((wb // 4,), float("nan"), device=d)
        g, loss = torch.full_like(p, float("nan")), torch.zeros(1, device=d)
        if tc:
            err = torch.zeros(1, dtype=torch.int32, device=d)
            P.ct_mlp_loss_grad_tc(p, Xt, Yt, Mt, n, g, loss, err, work, wb)
            assert int(err) == 0
        else:
            P.ct_mlp_loss_grad(p, Xt, Yt, Mt, n, g, loss, work, wb)
            out = torch.full((n, 10), float("nan"), device=d)
            P.ct_mlp_forward(p, Xt, n, out, work, wb)
            yref, _ = R.forward(theta.astype(np.float64), X.astype(np.float64))
            assert np.abs(out.cpu().numpy() - yref).max() <= 1e-4 * np.abs(yref).max()
        tol = (5e-2 if n == 1 else 1e-2) if tc else 1e-4
        assert float(loss) == pytest.approx(Lr, rel=tol)
        gg = g.cpu().numpy()
        assert np.linalg.norm(gg - gr) <= tol * np.linalg.norm(gr)


@pytest.mark.parametrize("n,batch", [(700, 128), (5000, 4097), (100, 200)])
def test_training_step_equals_gradient_and_adam(P, n, batch):
    """One epoch of ct_train_surrogate against the same steps taken with ct_mlp_loss_grad and
    ct_mlp_adam on the shuffled batches: the same kernels and order, so FP32 rounding apart
    (the compiler may fuse Adam differently) the parameters agree to 1e-5 of the step size."""
    X, Y, M = (torch.tensor(a, device="cuda") for a in _data(n, 3))
    theta = torch.tensor(_params(), device="cuda")
    p = theta.clone()
    stats = torch.zeros(4 * 26, device="cuda")
    wb = P.ct_train_workspace_bytes(n, batch, 1)
    work = torch.empty(wb // 4 + 64, device="cuda")
    lr = 1e-3
    cfg = dict(epochs=1, batch=batch, lr=lr, lr_final=lr, seed=9, tensor_cores=0, out_weight=[1.0] * 10)
    P.ct_train_surrogate(X, Y, M, n, cfg, p, stats, work, wb, torch.cuda.current_stream())
    s = stats.cpu()
    assert torch.allclose(s[:16], X.mean(0).cpu(), atol=1e-5)
    my = (Y * M).sum(0) / M.sum(0)
    assert torch.allclose(s[64:74], my.cpu(), atol=1e-5)
    perm, state, mask = list(range(n)), 9, (1 << 64) - 1
    for i in range(n - 1, 0, -1):
        state = (state + 0x9E3779B97F4A7C15) & mask
        z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        j = (z ^ (z >> 31)) % (i + 1)
        perm[i], perm[j] = perm[j], perm[i]
    sd = stats.view(-1)
    Xn = (X - sd[:16]) / sd[16:32]
    Yn = (Y - sd[64:74]) / sd[74:84] * M
    b = min(batch, n)
    q, m, v = theta.clone(), torch.zeros_like(theta), torch.zeros_like(theta)
    wb2 = P.ct_mlp_work_bytes(b)
    work2 = torch.empty(wb2 // 4 + 64, device="cuda")
    g, loss = torch.empty_like(q), torch.zeros(1, device="cuda")
    for k in range(n // b):
        idx = torch.tensor(perm[k * b:(k + 1) * b], device="cuda")
        P.ct_mlp_loss_grad(q, Xn[idx].contiguous(), Yn[idx].contiguous(), M[idx].contiguous(), b, g, loss, work2, wb2)
        P.ct_mlp_adam(q, g, m, v, q.numel(), lr, 0.9, 0.999, 1e-8, k + 1)
    assert float((p - q).norm()) <= 1e-3 * float((q - theta).norm())
