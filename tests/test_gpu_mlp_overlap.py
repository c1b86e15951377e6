"""Gradients written over the rows they are formed from: as with an array of their own, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 256, 3000])            # one chunk, and several
@pytest.mark.parametrize("over", ["x", "t"])
def test_gradient_over_its_rows(rows, over):
    import torch
    from paper_2307_00391_gb300.t0_model import T0Net
    gen = torch.Generator(device="cuda").manual_seed(rows)
    x, t = torch.randn((rows, 6), device="cuda", generator=gen), torch.randn((rows, 2), device="cuda", generator=gen)
    net = T0Net(params=T0Net.init_params(1))
    want, loss, loss2 = torch.empty(T0Net.N_PARAMS, device="cuda"), torch.empty(1, device="cuda"), torch.empty(1, device="cuda")
    net.gradients_dev(x, t, want, loss)
    src = x if over == "x" else t
    for shift in (0, 5):                                     # rows from the gradient's start, or a little inside
        pool = torch.zeros(max(src.numel() + shift, T0Net.N_PARAMS), device="cuda")
        rows_in = pool[shift:shift + src.numel()].view(src.shape)
        rows_in.copy_(src)
        grad = pool[:T0Net.N_PARAMS]
        net.gradients_dev(rows_in if over == "x" else x, rows_in if over == "t" else t, grad, loss2)
        assert torch.equal(grad, want) and torch.equal(loss, loss2)
    net.close()
