"""The loss of a long batch of one row repeated is that of four such rows, exactly: every partial loss is the
same FP32 value up to a power of two, and their FP64 sum rounds nothing away."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_rows", [3, 8, 13, 20])
def test_repeated_row(log_rows):
    import torch
    from paper_2307_00391_gb300.t0_model import T0Net
    gen = torch.Generator(device="cuda").manual_seed(log_rows)
    x, t = torch.randn((1, 6), device="cuda", generator=gen), torch.randn((1, 2), device="cuda", generator=gen)
    net = T0Net(params=T0Net.init_params(5))
    grad, loss, loss4 = torch.empty(T0Net.N_PARAMS, device="cuda"), torch.empty(1, device="cuda"), torch.empty(1, device="cuda")
    net.gradients_dev(x.expand(4, 6).contiguous(), t.expand(4, 2).contiguous(), grad, loss4)
    rows = 1 << log_rows
    net.gradients_dev(x.expand(rows, 6).contiguous(), t.expand(rows, 2).contiguous(), grad, loss)
    assert torch.equal(loss, loss4)
    net.close()
