"""The training pass at the edges of its split: one tile, fewer tiles than SMs, one CTA with several
tiles and a ragged last round, against the network with BF16 activations and deltas in FP64."""
import numpy as np
import pytest

from oracle import closure as cl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tv():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1004_5059_gb300 as tv
    return tv


def bf16_gradient(p, X, Ys):
    """Loss and gradient with every tensor-core operand rounded to BF16 (activations, g'(Z), deltas)."""
    r = cl.bf16_round
    Z1 = X @ p["W1"].T + p["b1"]
    H1, G1 = r(cl.gelu(Z1)), r(cl.gelu_grad(Z1))
    Z2 = H1 @ p["W2"].T + p["b2"]
    H2, G2 = r(cl.gelu(Z2)), r(cl.gelu_grad(Z2))
    D = H2 @ p["W3"].T + p["b3"] - Ys
    dY = 2.0 * D / D.size
    dZ2 = (r(dY) @ p["W3"]) * G2
    dZ1 = (r(dZ2) @ p["W2"]) * G1
    g = {"W3": r(dY).T @ H2, "b3": dY.sum(0), "W2": r(dZ2).T @ H1, "b2": dZ2.sum(0), "W1": r(dZ1).T @ X, "b1": dZ1.sum(0)}
    return float(np.mean(D ** 2)), g


# The reference rounds where the kernels do, so what differs is FP32 accumulation (relative 1e-6) and
# the few values that it pushes to the other side of a BF16 rounding (2^-8 of a value, in one value
# out of several thousand): 1e-3 of each gradient's norm.
@pytest.mark.parametrize("rows", [128, 1152, 128 * 152, 128 * 155, 128 * 333])
def test_gradient_matches_bf16_network(tv, rows):
    import torch
    rng = np.random.default_rng(rows)
    p = cl.init_params(41, scale=1.5)
    m = tv.Mlp(rows)
    m.set_params(cl.pack(p).astype(np.float32))
    X = np.zeros((rows, 64))
    X[:, :54] = cl.bf16_round(rng.normal(size=(rows, 54)))
    Y = np.zeros((rows, 16), dtype=np.float32)
    Y[:, :12] = rng.normal(size=(rows, 12)) * 0.5
    loss, grad = m.loss_grad(torch.from_numpy(X.astype(np.float32)).to(torch.bfloat16).cuda(), torch.from_numpy(Y).cuda(),
                             want_loss=True, want_grad=True)
    again, grad2 = m.loss_grad(torch.from_numpy(X.astype(np.float32)).to(torch.bfloat16).cuda(),
                               torch.from_numpy(Y).cuda(), want_loss=True, want_grad=True)
    assert loss == again and np.array_equal(grad, grad2)  # fixed summation orders
    pr = {k: cl.bf16_round(v) if k.startswith("W") else np.float32(v).astype(np.float64) for k, v in p.items()}
    L, g = bf16_gradient(pr, X[:, :54], Y[:, :12].astype(np.float64))
    assert abs(loss - L) <= 1e-4 * L
    for name, _ in cl.PARAM_SHAPES:
        a, b = cl.unpack(grad.astype(np.float64))[name].ravel(), g[name].ravel()
        assert np.linalg.norm(a - b) <= 1e-3 * np.linalg.norm(b), name
    m.close()
