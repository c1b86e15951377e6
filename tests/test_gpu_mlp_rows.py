"""The T0 network's row and gradient passes at the edges of their tiles (four rows per block, 1024
rows per gradient chunk) against the FP64 reference with the same BF16 weights.

Tolerance: FP32 sums of at most 128 terms of order 1 (forward) and of `rows` terms of order 1 / rows
(gradients): about 128 x 2^-24 = 8e-6 in the worst case, relative to the largest entry."""
import numpy as np
import pytest

from oracle import mlp_oracle as mo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 3, 4, 5, 129, 1023, 1024, 1025, 2050])
def test_rows(rows):
    import torch
    from paper_2307_00391_gb300.t0_model import T0Net
    rng = np.random.default_rng(rows)
    params = T0Net.init_params(rows)
    params[768:896] = rng.uniform(-0.1, 0.1, 128)          # biases too
    x = rng.standard_normal((rows, 6)).astype(np.float32)
    t = rng.standard_normal((rows, 2)).astype(np.float32)
    p64 = params.astype(np.float64)
    w = mo.unpack(p64)
    for name in ("W1", "W2", "W3"):
        w[name] = torch.tensor(w[name]).float().bfloat16().double().numpy()
    p64 = mo.pack(w)
    loss_ref, grad_ref = mo.loss_and_grad(p64, x, t)
    y_ref, _ = mo.forward(p64, x)
    net = T0Net(params=params)
    xd, td = torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda")
    y = torch.full((rows, 2), float("nan"), device="cuda")
    grad = torch.full((T0Net.N_PARAMS,), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), device="cuda")
    net.forward_dev(xd, y)
    net.gradients_dev(xd, td, grad, loss)
    tol = 1e-5
    assert np.abs(y.cpu().numpy() - y_ref).max() <= tol * np.abs(y_ref).max()
    g = grad.cpu().numpy()
    for name, (a, b) in zip([s[0] for s in mo.SIZES], zip(np.cumsum([0] + [int(np.prod(s[1])) for s in mo.SIZES])[:-1],
                                                         np.cumsum([int(np.prod(s[1])) for s in mo.SIZES]))):
        assert np.abs(g[a:b] - grad_ref[a:b]).max() <= tol * np.abs(grad_ref[a:b]).max(), name
    assert float(loss) == pytest.approx(loss_ref, rel=tol)
    net.close()
