"""Measurements of one state on two streams at once with one plan: whatever they give, the ticket counter that
picks the last block is back at zero afterwards, so the next measurement is complete."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["c64", "c128"])
def test_counter_returns_to_zero(precision):
    import torch
    import paper_2307_00391_gb300 as hhl
    n_s, n_c = 8, 8
    n = 1 << n_s
    diag, off = hhl.laplacian(n)
    plan = hhl.HHLPlan(n_s, n_c, diag=diag, off=off, precision=precision)
    state = plan.new_state()
    plan.prepare_rhs(torch.ones(n, dtype=torch.complex128, device="cuda"), state)
    want, got = (torch.full((4 + 2 * n,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
    plan.measure_async(state, want)
    side = [torch.cuda.Stream() for _ in range(2)]
    outs = [torch.empty_like(want) for _ in side]
    torch.cuda.synchronize()
    for _ in range(100):
        for s, o in zip(side, outs):
            plan.measure_async(state, o, stream=s)
    torch.cuda.synchronize()
    plan.measure_async(state, got)
    assert torch.equal(got, want)
    plan.close()
