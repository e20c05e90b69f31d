"""The tensor-core training loop, whose reduction also rewrites both BF16 operand orders of the
weights, against the same batches taken with ct_mlp_loss_grad_tc (which packs them anew from the FP32
parameters) and ct_mlp_adam."""
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


# The kernels, rows and order are the same; FP32 roundings of the standardised rows and of Adam, which
# the compiler may fuse differently, may flip single BF16 roundings.  Bound: 1 % of the parameters'
# movement (operands that stay as they were before the first step move it by 10 to 14 %).
@pytest.mark.parametrize("n,batch", [(700, 128), (2700, 300), (4100, 1300)])
def test_training_steps_equal_gradients_and_adam(P, n, batch):
    rng = np.random.default_rng(3)
    X, Y, M = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in
               (rng.standard_normal((n, 16)), rng.standard_normal((n, 10)), rng.uniform(size=(n, 10)) > 0.25))
    theta = torch.tensor(R.init_params(3) + 0.01 * np.random.default_rng(5).standard_normal(R.n_params()), dtype=torch.float32, device="cuda")
    p = theta.clone()
    stats = torch.zeros(4 * 26, device="cuda")
    wb = P.ct_train_workspace_bytes(n, batch, 1)
    work = torch.empty(wb // 4 + 64, device="cuda")
    lr = 3e-3
    cfg = dict(epochs=1, batch=batch, lr=lr, lr_final=lr, seed=9, tensor_cores=1, out_weight=[1.0] * 10)
    P.ct_train_surrogate(X, Y, M, n, cfg, p, stats, work, wb, torch.cuda.current_stream())
    perm, state, mask = list(range(n)), 9, (1 << 64) - 1
    for i in range(n - 1, 0, -1):
        state = (state + 0x9E3779B97F4A7C15) & mask
        z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        j = (z ^ (z >> 31)) % (i + 1)
        perm[i], perm[j] = perm[j], perm[i]
    Xn = (X - stats[:16]) / stats[16:32]
    Yn = (Y - stats[64:74]) / stats[74:84] * M
    q, m, v = theta.clone(), torch.zeros_like(theta), torch.zeros_like(theta)
    wb2 = P.ct_mlp_work_bytes(batch)
    work2 = torch.empty(wb2 // 4 + 64, device="cuda")
    g, loss, err = torch.empty_like(q), torch.zeros(1, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    for k in range(n // batch):
        idx = torch.tensor(perm[k * batch:(k + 1) * batch], device="cuda")
        P.ct_mlp_loss_grad_tc(q, Xn[idx].contiguous(), Yn[idx].contiguous(), M[idx].contiguous(), batch, g, loss, err, work2, wb2)
        P.ct_mlp_adam(q, g, m, v, q.numel(), lr, 0.9, 0.999, 1e-8, k + 1)
    assert int(err) == 0
    assert float((p - q).norm()) <= 1e-2 * float((q - theta).norm())
