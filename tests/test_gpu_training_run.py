"""A training run of the closure network: iterations of gradient and Adam step, each from the parameters
that the one before left, against the BF16 network in FP64 arithmetic with the same Adam steps."""
import numpy as np
import pytest

from oracle import closure as cl
from test_gpu_closure_train import bf16_gradient

pytestmark = pytest.mark.gpu

LR, BETA1, BETA2, EPS, ITERS = 1e-3, 0.9, 0.999, 1e-8, 8


@pytest.fixture(scope="module")
def tv():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1004_5059_gb300 as tv
    return tv


def batches(rows):
    rng = np.random.default_rng(rows + 1)
    X = np.zeros((ITERS, rows, 64))
    X[:, :, :54] = cl.bf16_round(rng.normal(size=(ITERS, rows, 54)))
    t = rng.normal(size=(54, 12)) / np.sqrt(54.0)
    Y = np.zeros((ITERS, rows, 16), dtype=np.float32)
    Y[:, :, :12] = np.tanh(X[:, :, :54] @ t)
    return X, Y


def run(tv, theta, X, Y):
    import torch
    m = tv.Mlp(X.shape[1])
    m.set_params(theta)
    x = torch.from_numpy(X.astype(np.float32)).to(torch.bfloat16).cuda()
    y = torch.from_numpy(Y).cuda()
    for k in range(ITERS):
        grad = m.loss_grad(x[k], y[k], want_loss=False, want_grad=k == ITERS - 1)[1]
        m.adam(LR, BETA1, BETA2, EPS)
    out = grad, m.get_params()
    m.close()
    return out


# Each iteration's gradient may be 1e-3 of its norm off (the bound of a single pass, see
# test_gpu_closure_train), and what an iteration adds is carried on: 8e-3 after eight.  Adam's first steps
# have the size of the learning rate whatever the gradient's, so a parameter whose gradient lies within
# its error may step the wrong way: at 1e-3 of the norm that is one in 1200, 2 sqrt(1 / 1200) = 6e-2 of the
# norm of the way gone.  8320 rows: beyond the batches whose partial sums are 64 rows each.
@pytest.mark.parametrize("rows", [1024, 8320])
def test_training_run_follows_the_bf16_network(tv, rows):
    X, Y = batches(rows)
    theta0 = cl.pack(cl.init_params(43, scale=1.0)).astype(np.float32)
    grad, theta = run(tv, theta0, X, Y)
    grad2, theta2 = run(tv, theta0, X, Y)
    assert np.array_equal(grad, grad2) and np.array_equal(theta, theta2)  # fixed summation orders
    th, m1, m2 = theta0.astype(np.float64), 0.0, 0.0
    for k in range(ITERS):
        p = {n: cl.bf16_round(v) if n.startswith("W") else v for n, v in cl.unpack(th).items()}
        g = cl.pack(bf16_gradient(p, X[k, :, :54], Y[k, :, :12].astype(np.float64))[1])
        m1, m2 = BETA1 * m1 + (1 - BETA1) * g, BETA2 * m2 + (1 - BETA2) * g * g
        step = LR * (m1 / (1 - BETA1 ** (k + 1))) / (np.sqrt(m2 / (1 - BETA2 ** (k + 1))) + EPS)
        th = (th - step).astype(np.float32).astype(np.float64)  # the parameters are FP32
    assert np.linalg.norm(grad - g) <= 8e-3 * np.linalg.norm(g)
    assert np.linalg.norm(theta - th) <= 6e-2 * np.linalg.norm(th - theta0)


def test_activation_does_not_depend_on_the_place_in_a_pair(tv):
    """Entries are taken in pairs: an entry first, second or alone in its pair gives the same bits."""
    import torch
    z = torch.linspace(-9.0, 9.0, 4097, dtype=torch.float32, device="cuda")
    g, dg = tv.mlp_activation(z)
    g1, dg1 = tv.mlp_activation(z[1:].clone())  # every entry in the other place, an even number of them
    assert torch.equal(g[1:], g1) and torch.equal(dg[1:], dg1)
    g2, dg2 = tv.mlp_activation(z[2048:2049].clone())
    assert g2.item() == g[2048].item() and dg2.item() == dg[2048].item()
