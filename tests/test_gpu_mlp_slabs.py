"""Batches of more rows than the activation buffers hold: the chunks' gradients (1024 rows each) are added in
row order whatever the slab, so a batch of 2^19 rows gives exactly the FP32 sum of its 512 chunks' gradients,
each computed alone (the loss's 1 / rows is a power of two either way)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_rows", [11, 18, 19])
def test_sum_of_the_chunks(log_rows):
    import torch
    from paper_2307_00391_gb300.t0_model import T0Net
    rows, chunk = 1 << log_rows, 1024
    gen = torch.Generator(device="cuda").manual_seed(log_rows)
    x = torch.randn((rows, 6), device="cuda", generator=gen)
    t = torch.randn((rows, 2), device="cuda", generator=gen)
    net = T0Net(params=T0Net.init_params(3))
    grad, part = (torch.empty(T0Net.N_PARAMS, device="cuda") for _ in range(2))
    loss, loss1 = (torch.empty(1, device="cuda") for _ in range(2))
    net.gradients_dev(x, t, grad, loss)
    total, mean = None, 0.0
    for r in range(0, rows, chunk):
        net.gradients_dev(x[r:r + chunk], t[r:r + chunk], part, loss1)
        g = part * (chunk / rows)
        total = g if total is None else total + g
        mean += float(loss1) * chunk / rows
    assert torch.equal(grad, total)
    assert float(loss) == pytest.approx(mean, rel=3e-4)   # 2^12 FP32 terms a lane: 2^12 x 2^-24 at worst
    net.close()
