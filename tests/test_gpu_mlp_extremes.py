"""The training kernels' SiLU at the ends of FP32, as z / (1 + exp(-z)) has it: a pre-activation that
overflows keeps its infinity, and one near -86, where 1 + exp(-z) exceeds 1e37, keeps its slope."""
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


@pytest.mark.parametrize("n", [5, 3000])      # tiles of 32 rows and of 64
def test_an_overflowing_activation_stays_infinite(P, n):
    theta = torch.ones(R.n_params(), device="cuda")       # every product positive: +inf all the way
    X = torch.full((n, 16), 3e38, device="cuda")
    Y = torch.zeros(n, 10, device="cuda")
    wb = P.ct_mlp_work_bytes(n)
    P.ct_mlp_forward(theta, X, n, Y, torch.empty(wb // 4, device="cuda"), wb)
    assert torch.isposinf(Y).all()


# The first layer's unit 0 has z = x_0 - 86.2; the weights behind it bring its value, about -86 e^-86,
# back to order one.  Everything else is zero.  __expf(86) carries some 100 ulp (1e-5); BF16 operands 2^-9 each
# over eight products.
@pytest.mark.parametrize("n", [40, 3000])
@pytest.mark.parametrize("tc", [False, True])
def test_slope_of_a_deeply_negative_activation(P, n, tc):
    theta = np.zeros(R.n_params(), dtype=np.float32)
    layers = R.unpack(theta)                              # views into theta
    for l in range(5):
        layers[l][0][:, 0] = 1.0 if l == 4 else 0.0
        layers[l][0][0, 0] = 1.0
    layers[0][1][0] = -86.2
    layers[1][0][0, 0] = 1e35
    assert theta[0] == 1.0
    rng = np.random.default_rng(4)
    X = np.zeros((n, 16), dtype=np.float32)
    X[:, :4] = rng.uniform(-0.5, 0.5, (n, 4))
    Y = rng.uniform(1.0, 2.0, (n, 10)).astype(np.float32)
    M = np.ones((n, 10), dtype=np.float32)
    _, gr = R.loss_and_grad(theta.astype(np.float64), X.astype(np.float64), Y.astype(np.float64), M.astype(np.float64))
    t = lambda a: torch.tensor(a, device="cuda")
    wb = P.ct_mlp_work_bytes(n)
    work = torch.empty(wb // 4, device="cuda")
    g, loss, err = torch.empty(theta.size, device="cuda"), torch.zeros(1, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    if tc:
        P.ct_mlp_loss_grad_tc(t(theta), t(X), t(Y), t(M), n, g, loss, err, work, wb)
        assert int(err) == 0
    else:
        P.ct_mlp_loss_grad(t(theta), t(X), t(Y), t(M), n, g, loss, work, wb)
    b0 = 128 * 16                                         # the first layer's bias of unit 0
    got, ref = g.cpu().numpy()[[0, 1, 2, 3, b0]], gr[[0, 1, 2, 3, b0]]
    assert abs(ref[4]) > 1e-4
    assert np.linalg.norm(got - ref) <= (5e-2 if tc else 1e-3) * np.linalg.norm(ref)
